// Time-interval policies, a thread per policy (sm_100a): emo_walk walks the walk program of emo_walk.h.
// Included only by emo_lib.cu.
//
// A start decides a level, a level a duration, a duration the next start: the chain of Alg. 1 runs through every node, and what a
// thread keeps of it is the current interval: how much of it is left, where its level lies in a table row, and the next
// interval's.  An item of up to eight nodes is then eight loads, their running sums and one comparison of the last with what is
// left.  Where some policy of the warp leaves its interval, the boundary falls behind a node that the sums already show: the nodes
// behind it are loaded again at the next level; only where a node outlasts a whole interval are they taken one by one.
// Busy time is kept per thread while the (row, interval) stays the same and added to busy[row][interval][policy] when it changes.
//
// What bounds it: one warp's latencies, about 150 cycles an item and 360 more where it has nodes; the time of a call hardly depends on
// the policies as long as a block's warps cover them (25 000 nodes: 1.63 ms for 16, 1.68 for 16 384).  The lane-stream kernel, a warp
// per lane of the schedule, is faster where it has many lanes (there, five, 0.90 and 1.05 ms), this one where it has few or where
// its blocks come in several waves (see walk_pays).
#pragma once
#include "emo_flow.cuh"
#include "emo_walk.h"

constexpr int kWalkBig = (1 << 30) - 1;          // what is left of the last interval, renewed when used up
constexpr int kWalkMaxBuffers = 4;
constexpr int kWalkMaxGroups = 12;               // most warps of a block that walk

struct WalkParams {
    const unsigned char *blob;
    int chunks, buffers, Lp, L;
    unsigned chunk_bytes, off_dur, off_en;
    int groups, pl, P;                   // warps that walk; policies of each, of the block
    unsigned off_F, off_slots, off_buf;  // shared memory (the barriers come first)
    int rows, I;
    int64_t B;
    const uint8_t *F;
    int64_t ldF;
    int delta;                           // length of an interval
    float inv;                           // 1 / delta
    double energy0;
    int64_t *makespan;
    double *energy;
    unsigned long long *busy;            // or null
    int64_t ldw;
    int32_t *status;
    long long wait_cycles;
};

__device__ __forceinline__ long long emo_walk_ld64(unsigned a)
{
    long long v;
    asm volatile("ld.shared.b64 %0, [%1];" : "=l"(v) : "r"(a));
    return v;
}
__device__ __forceinline__ double emo_walk_ldf(unsigned a)
{
    double v;
    asm volatile("ld.shared.f64 %0, [%1];" : "=d"(v) : "r"(a));
    return v;
}
// the word at a where `take`, else zero
__device__ __forceinline__ unsigned emo_walk_ld_if(unsigned a, bool take)
{
    unsigned v;
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %2, 0;\n\tmov.u32 %0, 0;\n\t@p ld.shared.u32 %0, [%1];\n\t}" : "=r"(v) : "r"(a), "r"((unsigned)take));
    return v;
}
__device__ __forceinline__ double emo_walk_ldf_if(unsigned a, bool take)
{
    double v;
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %2, 0;\n\tmov.f64 %0, 0d0000000000000000;\n\t@p ld.shared.f64 %0, [%1];\n\t}" : "=d"(v) : "r"(a), "r"((unsigned)take));
    return v;
}

// A thread's place in its policy.
struct WalkState {
    long long iend;                      // end of the current interval (the last one: a time not yet reached)
    long long bacc;                      // busy time in it that is not yet in memory
    int left, i, row;                    // iend - now, > 0 between items; interval; its policy row
    unsigned la, la2;                    // its level and the next interval's, as offsets into a row of durations
    double E;
    unsigned f_a;                        // this policy's level of row 0, interval 0
    unsigned long long *busy;            // [rows][I], ldw apart; null: not wanted or no such policy

    __device__ __forceinline__ unsigned level(const WalkParams &p, int r, int k) const
    {
        return 4u * emo_lds_u8(f_a + (unsigned)(r * p.I + k) * (unsigned)p.P);
    }
    __device__ __forceinline__ void flush(const WalkParams &p, long long t)
    {
        if (busy && t) atomicAdd(busy + (size_t)(row * p.I + i) * p.ldw, (unsigned long long)t);
    }
    // the interval that holds t, of policy row r
    __device__ __forceinline__ void look_up(const WalkParams &p, long long t, int r)
    {
        int k = min((int)(__ll2float_rz(t) * p.inv), p.I - 1);
        long long lo = (long long)k * p.delta;
        // (the guess is off by one at most: 4 096 intervals against 2^-23)
        if (t < lo) {
            --k;
            lo -= p.delta;
        } else if (k < p.I - 1 && t >= lo + p.delta) {
            ++k;
            lo += p.delta;
        }
        if (k != i || r != row) {
            flush(p, bacc);
            bacc = 0;
        }
        i = k;
        row = r;
        la = level(p, r, k);
        la2 = level(p, r, min(k + 1, p.I - 1));
        if (k == p.I - 1) {
            left = kWalkBig;
            iend = t + kWalkBig;
        } else {
            iend = lo + p.delta;
            left = (int)(iend - t);
        }
    }
    // into the next interval, `over` behind its beginning
    __device__ __forceinline__ void advance(const WalkParams &p, int over)
    {
        const int k = min(i + 1, p.I - 1), step = k == p.I - 1 ? kWalkBig : p.delta;
        i = k;
        iend += step;
        left = step - over;
        la = la2;
        la2 = level(p, row, min(k + 1, p.I - 1));
    }
    // n <= K nodes, durations from da on, energies from ea on
    template <int K>
    __device__ __forceinline__ void run(const WalkParams &p, int n, unsigned da, unsigned ea)
    {
        const unsigned rb = (unsigned)p.Lp * 4u;
        unsigned at[K], s[K];
#pragma unroll
        for (int j = 0; j < K; ++j) {
            at[j] = da + (unsigned)j * rb + la;
            s[j] = emo_walk_ld_if(at[j], j < n);
        }
#pragma unroll
        for (int j = 1; j < K; ++j) s[j] += s[j - 1];
        if (!__any_sync(0xFFFFFFFFu, (int)s[K - 1] >= left)) {
            left -= (int)s[K - 1];
            bacc += s[K - 1];
        } else {
            // nodes that start at or behind the boundary: the next interval's level
            const bool leaves = (int)s[K - 1] >= left;
            const unsigned d = la2 - la;
            unsigned sum = s[0];
#pragma unroll
            for (int j = 1; j < K; ++j) {
                if ((int)s[j - 1] >= left) at[j] += d;
                sum += emo_walk_ld_if(at[j], j < n);
            }
            const int over = leaves ? (int)sum - left : 0;
            const int step = i + 1 >= p.I - 1 ? kWalkBig : p.delta;
            if (__any_sync(0xFFFFFFFFu, over >= step)) {
                one_by_one<K>(p, n, da, ea);
                return;
            }
            if (leaves) {
                flush(p, bacc + left);
                bacc = over;
                advance(p, over);
            } else {
                left -= (int)sum;
                bacc += sum;
            }
        }
        double e[K];
#pragma unroll
        for (int j = 0; j < K; ++j) e[j] = emo_walk_ldf_if(ea + 2u * (at[j] - da), j < n);
#pragma unroll
        for (int w = 1; w < K; w *= 2)
#pragma unroll
            for (int j = 0; j + w < K; j += 2 * w) e[j] += e[j + w];
        E += e[0];
    }
    // The same node after node, where some policy of the warp has a node that outlasts an interval.  The energies are added pair by pair as
    // above: a policy's energy does not depend on the policies beside it.
    template <int K>
    __device__ __forceinline__ void one_by_one(const WalkParams &p, int n, unsigned da, unsigned ea)
    {
        double one = 0.0, two = 0.0, four = 0.0, sum = 0.0;      // first halves of the pairs, of the fours, of the eight
#pragma unroll 1
        for (int j = 0; j < K; ++j) {
            double e = 0.0;
            if (j < n) {
                const unsigned o = (unsigned)j * (unsigned)p.Lp * 4u + la;
                const int d = (int)emo_lds_u32(da + o);
                e = emo_walk_ldf(ea + 2u * o);
                bacc += d;
                left -= d;
                while (left <= 0) {
                    flush(p, bacc + left);
                    bacc = -left;
                    advance(p, -left);
                }
            }
            if (!(j & 1)) {
                one = e;
            } else if (!(j & 2)) {
                two = one + e;
            } else if (!(j & 4)) {
                sum = four = two + (one + e);
            } else {
                sum = four + (two + (one + e));
            }
        }
        E += sum;
    }
};

__global__ void __launch_bounds__((kWalkMaxGroups + 1) * 32, 1) emo_walk(WalkParams p)
{
    extern __shared__ __align__(128) unsigned char emo_smem[];
    const unsigned smem0 = emo_smem_addr(emo_smem);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    volatile int *const abort_word = reinterpret_cast<volatile int *>(emo_smem + 2 * kWalkMaxBuffers * 8);
    const int64_t b0 = (int64_t)blockIdx.x * p.P;
    const unsigned full0 = smem0, empty0 = smem0 + kWalkMaxBuffers * 8;
    if (threadIdx.x == 0) {
        for (int k = 0; k < p.buffers; ++k) {
            emo_mbar_init(full0 + 8u * k, 1);
            emo_mbar_init(empty0 + 8u * k, (unsigned)p.groups);
        }
        abort_word[0] = 0;
        abort_word[1] = 0;               // never set: the drain after a failure waits its full time
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    // the block's columns of the levels; slot 0 is the time zero
    for (int k = threadIdx.x; k < p.rows * p.I * p.P; k += blockDim.x) {
        const int64_t b = b0 + k % p.P;
        unsigned f = b < p.B ? p.F[(int64_t)(k / p.P) * p.ldF + b] : 0u;
        emo_smem[p.off_F + k] = (unsigned char)(f & ((unsigned)p.Lp - 1u));
    }
    for (int k = threadIdx.x; k < p.groups * 32; k += blockDim.x) reinterpret_cast<long long *>(emo_smem + p.off_slots)[k] = 0;
    __syncthreads();
    if (warp == p.groups) {
        // the producer: one bulk copy per chunk
        if (lane != 0) return;
        int k = 0;
        for (; k < p.chunks; ++k) {
            const int s = k % p.buffers;
            if (k >= p.buffers && !emo_spine_wait(empty0 + 8u * s, ((k / p.buffers) & 1) ^ 1, abort_word, p.wait_cycles)) {
                *abort_word = 1;
                if (p.status) atomicMin(p.status, -8);
                break;
            }
            emo_mbar_expect_tx(full0 + 8u * s, p.chunk_bytes);
            emo_bulk_g2s(smem0 + p.off_buf + (unsigned)s * p.chunk_bytes, p.blob + (size_t)k * p.chunk_bytes, p.chunk_bytes, full0 + 8u * s);
        }
        // not before the copies have landed, whatever the other warps do
        for (int c = max(0, k - p.buffers); c < k; ++c)
            (void)emo_spine_wait(full0 + 8u * (c % p.buffers), (c / p.buffers) & 1, abort_word + 1, max(p.wait_cycles, 20000000LL));
        return;
    }
    // (lanes behind the warp's policies walk along with copies of them)
    const int col = warp * p.pl + lane % p.pl;
    const int64_t b = b0 + col;
    const bool mine = lane < p.pl && b < p.B;
    WalkState w;
    w.iend = w.bacc = 0;
    w.left = 1;
    w.i = w.row = 0;
    w.la = w.la2 = 0;
    w.E = 0.0;
    w.f_a = smem0 + p.off_F + (unsigned)col;
    w.busy = mine && p.busy ? p.busy + b : nullptr;
    const unsigned slot_pitch = (unsigned)p.groups * 256u, slots = smem0 + p.off_slots + (unsigned)warp * 256u + (unsigned)lane * 8u;
    long long t = 0, T = 0;
    for (int k = 0; k < p.chunks; ++k) {
        const int s = k % p.buffers;
        if (!emo_spine_wait(full0 + 8u * s, (k / p.buffers) & 1, abort_word, p.wait_cycles)) {
            if (lane == 0) {
                *abort_word = 1;
                if (p.status) atomicMin(p.status, -8);
            }
            return;
        }
        const unsigned buf = smem0 + p.off_buf + (unsigned)s * p.chunk_bytes, dur = buf + p.off_dur, en = buf + p.off_en;
        const unsigned rb = (unsigned)p.Lp * 4u;
        const unsigned items = emo_lds_u32(buf);
        unsigned at = buf + 16u;
        uint4 it = emo_lds128(at);
        for (unsigned q = 0; q < items; ++q) {
            const uint4 c = it;
            at += 16u;
            it = emo_lds128(at);             // (behind the last: a spare one)
            if (c.x & emo::kWalkStart) {
                const long long x = emo_walk_ld64(slots + (c.y & 0xFFFFu) * slot_pitch), y = emo_walk_ld64(slots + (c.y >> 16) * slot_pitch);
                const long long z = max(x, y);
                t = (c.x & emo::kWalkMore) ? max(t, z) : z;
            }
            if (c.x & emo::kWalkFix) t += c.z;
            const int n = (int)(c.x & 15u);
            if (n) {
                if (c.x & emo::kWalkFresh) w.look_up(p, t, (int)c.z);
                const unsigned da = dur + c.w * rb, ea = en + c.w * rb * 2u;
                if (n <= 4) w.run<4>(p, n, da, ea);
                else w.run<8>(p, n, da, ea);
                t = w.iend - w.left;
            }
            if (c.x & emo::kWalkPub) asm volatile("st.shared.b64 [%0], %1;" ::"r"(slots + (c.x >> 16) * slot_pitch), "l"(t) : "memory");
            if (c.x & emo::kWalkTerm) T = max(T, t);
        }
        __syncwarp();
        if (lane == 0) emo_mbar_arrive(empty0 + 8u * s);
    }
    w.flush(p, w.bacc);
    if (mine) {
        p.makespan[b] = T;
        p.energy[b] = w.E + p.energy0;
    }
}
