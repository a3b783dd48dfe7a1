// The slice kernels (sm_100a): calls with few policies, all slices of the graph at once (see emo_slice.h).
// Included only by emo_lib.cu.
//
//   emo_slice_matrix   per slice and tile of P policies: durations, running sums along the paths, then per policy and direction the
//                      slice's matrix, a thread per column: the values of all operations with that column's value at zero and the
//                      others absent; also the slice's energy
//   emo_slice_group    (many slices) products of a group's matrices
//   emo_slice_scan     chains matrices with vectors: the values that enter every slice, the makespan, the energy
//   emo_slice_whole    all of it in one block per policy where the graph is a few slices
//   emo_slice_values   per slice and tile: running sums again, every operation once with the values that enter, then ES, LS, slack of
//                      every node; alone where the graph is one slice
// Only `values` writes per node and policy; a forward-only call ends with `scan`.
//
// A thread works on values of its own (one policy, one column), so the operations need no synchronisation; what bounds a call is
// the chain of a slice's steps (a shared load, an addition, two maxima, a store that the next step may read) and the kernels'
// first loads, with more policies the issue slots of the columns.  Slices are short because the chain is; they are chained in two
// levels because otherwise chaining would take longer than they do.  Measured (us a call, slack, spine kernels / these): 250 000 nodes
// x 1 policy 8 720 / 80, 10 000 x 1 593 / 31, 1 013 x 1 86 / 19, 400 x 64 31 / 17, 250 000 x 256 7 416 / 1 749, 10 000 x 1 024 596 / 348.
#pragma once
#include "emo_flow.cuh"
#include "emo_slice.h"

using emo::SliceHdr;

constexpr int kSliceNone32 = -(1 << 30);         // no path (stays negative with any path of a slice or group added)

struct SliceParams {
    const uint32_t *blob;                // programs of the slices
    const uint4 *index;                  // [count] first word, nodes, the first one's place, words of header, paths and rows | all words << 16
    const uint4 *rec;                    // [n] see Slices
    const uint32_t *tabT;                // [n][Lp]
    const double *tabE;                  // [n][Lp]
    int count, cols, Lp, L, dirs;        // dirs: 1 forward only, 2 both
    int group, groups;
    int tiles;
    unsigned at_rec, at_ops[2], at_inc[2], at_slot[2];      // shared memory of a slice (bytes)
    unsigned slice_bytes, at_red;        // ... of all of a slice; behind the block's slices
    int64_t B, nb, nbp;                  // policies, with the virtual all-max one (column B), rounded up to whole tiles
    const uint8_t *lvl;
    int64_t ldb;
    int32_t *mat[2];                     // [count][nbp][cols][cols]: row, column
    int32_t *gmat[2];                    // [groups][nbp][cols][cols]
    long long *state[2];                 // [count][nbp][cols] values that enter a slice
    double *epart, *gepart;              // [count][nbp] energies of the slices, [groups][nbp] of the groups
    int64_t *makespan;
    double *energy;
    int64_t *base_T;
    double *base_E;
    int64_t *ES, *LS, *slack;
    int64_t ldo;
    int64_t *slack_sum;
    int32_t *n_critical;
};

// Header, paths and rows of a slice's program to shared memory, 16 bytes at a time.
template <int T>
__device__ __forceinline__ void emo_slice_stage(uint32_t *dst, const uint32_t *src, unsigned words, int tid)
{
    for (unsigned i = tid; i < words / 4; i += T) reinterpret_cast<uint4 *>(dst)[i] = __ldg(reinterpret_cast<const uint4 *>(src) + i);
}
// Steps of a slice and direction to shared memory, slots and entries as byte offsets: a thread then adds what is its own to each.
// One more (of zeros) is read ahead.
template <int T>
__device__ __forceinline__ void emo_slice_steps(unsigned char *dst, const uint32_t *src, unsigned steps, unsigned slot_bytes, unsigned entry_bytes, int tid)
{
    for (unsigned i = tid; i <= steps; i += T) {
        const uint4 w = __ldg(reinterpret_cast<const uint4 *>(src) + i);      // two operands, slot to write, whether it is the operation's last
        reinterpret_cast<uint4 *>(dst + i * 32u)[0] = make_uint4((w.x & 0xFFFFu) * slot_bytes, (w.x >> 16) * entry_bytes, (w.y & 0xFFFFu) * slot_bytes, (w.y >> 16) * entry_bytes);
        reinterpret_cast<uint2 *>(dst + i * 32u)[2] = make_uint2(w.z * slot_bytes, w.w);
    }
}

// Durations of all nodes of a slice for this thread's policy into the entries of the running sums, and their energies.
template <int P, int T, bool ENERGY>
__device__ __forceinline__ double emo_slice_look(const SliceParams &p, const SliceHdr &h, const uint4 *rec, uint32_t *incF, uint32_t *incB, int64_t b, int tid)
{
    constexpr int U = 4, STEP = T / P;
    const int pl = tid % P, n = (int)h.nodes;
    const bool both = p.dirs > 1;
    const uint8_t *const col = p.lvl + b;
    const unsigned mask = (unsigned)p.Lp - 1u, fixed = b == p.B ? (unsigned)(p.L - 1) : 0u;
    const bool read = b < p.B;
    const uint32_t *const lat = p.tabT + (size_t)h.node0 * p.Lp;
    const double *const E = p.tabE + (size_t)h.node0 * p.Lp;
    double ea = 0.0;
    for (int i0 = tid / P; i0 < n; i0 += U * STEP) {
        uint4 r[U];
        unsigned lv[U], d[U];
        double e[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            r[u] = rec[min(i0 + u * STEP, n - 1)];
            lv[u] = 0u;
            if (r[u].x != emo::kNone) lv[u] = read ? (unsigned)__ldcg(col + (int64_t)r[u].x * p.ldb) & mask : fixed;
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const unsigned at = (unsigned)min(i0 + u * STEP, n - 1) * (unsigned)p.Lp + lv[u];
            d[u] = __ldg(lat + at);
            if (ENERGY) e[u] = __ldg(E + at);
        }
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (i0 + u * STEP < n) {
                incF[(r[u].z & 0xFFFFu) * P + pl] = d[u];
                if (both) incB[(r[u].z >> 16) * P + pl] = d[u];
                if (ENERGY) ea += e[u];
            }
    }
    return ea;
}

// Running sums along the paths, a thread per path and policy.
template <int P, int T>
__device__ __forceinline__ void emo_slice_sums(const SliceHdr &h, const uint32_t *prog, uint32_t *incF, uint32_t *incB, int dirs, int tid)
{
    const int pl = tid % P, nf = (int)h.dir[0].paths, total = nf + (dirs > 1 ? (int)h.dir[1].paths : 0);
    for (int t = tid / P; t < total; t += T / P) {
        const bool fwd = t < nf;
        const uint32_t w = fwd ? prog[h.dir[0].off_path + t] : prog[h.dir[1].off_path + t - nf];
        uint32_t *a = (fwd ? incF : incB) + (w & 0xFFFFu) * P + pl;
        const int len = (int)(w >> 16);
        uint32_t run = 0;
        a[0] = 0;
        int i = 1;
        for (; i + 3 <= len; i += 4) {
            const uint32_t d0 = a[i * P], d1 = a[(i + 1) * P], d2 = a[(i + 2) * P], d3 = a[(i + 3) * P];
            a[i * P] = run += d0;
            a[(i + 1) * P] = run += d1;
            a[(i + 2) * P] = run += d2;
            a[(i + 3) * P] = run += d3;
        }
        for (; i <= len; ++i) a[i * P] = run += a[i * P];
    }
}

__device__ __forceinline__ void emo_slice_ld(int &v, unsigned a) { asm volatile("ld.shared.b32 %0, [%1];" : "=r"(v) : "r"(a)); }
__device__ __forceinline__ void emo_slice_ld(long long &v, unsigned a) { asm volatile("ld.shared.b64 %0, [%1];" : "=l"(v) : "r"(a)); }
__device__ __forceinline__ void emo_slice_st(unsigned a, int v) { asm volatile("st.shared.b32 [%0], %1;" ::"r"(a), "r"(v) : "memory"); }
__device__ __forceinline__ void emo_slice_st(unsigned a, long long v) { asm volatile("st.shared.b64 [%0], %1;" ::"r"(a), "l"(v) : "memory"); }

// The operations of a slice and direction for this thread's values (its word of slot 0 at vals, of entry 0 at inc), two operands a
// step; what an operation has so far stays in a register (a step that is not its last writes a slot nobody reads).  (Steps of two
// independent operations, or four operands, had half of their operands empty on graphs with serial chains: 10 000 nodes x 1 024
// policies 0.41 ms.)
template <typename V>
__device__ __forceinline__ void emo_slice_ops(unsigned at, unsigned steps, unsigned vals, unsigned inc)
{
    const V none = (V)kSliceNone32;
    V acc = none;
    uint4 a = emo_lds128(at);
    uint2 d;
    asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(d.x), "=r"(d.y) : "r"(at + 16u));
    for (unsigned k = 0; k < steps; ++k) {
        V x0, x1;
        int s0, s1;
        emo_slice_ld(x0, vals + a.x);
        emo_slice_ld(x1, vals + a.z);
        emo_slice_ld(s0, inc + a.y);
        emo_slice_ld(s1, inc + a.w);
        const unsigned to = vals + d.x, last = d.y;
        at += 32u;
        a = emo_lds128(at);              // (behind the last: a spare one)
        asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(d.x), "=r"(d.y) : "r"(at + 16u));
        const V y = max(max(acc, x0 + (V)(unsigned)s0), x1 + (V)(unsigned)s1);
        emo_slice_st(to, y);
        acc = last ? none : y;
    }
}

// P policies by S slices per block of NT threads, NT / S of them on a slice; the operations of all of them side by side in the lanes
// of a warp.  (One policy alone has a column in 6 lanes of 32, and the shared-memory pipe takes as long for them as for 32: four
// slices share a warp.)
template <int P, int S, int NT>
__global__ void __launch_bounds__(NT) emo_slice_matrix(SliceParams p)
{
    extern __shared__ __align__(128) unsigned char emo_smem[];
    constexpr int T = NT / S;
    const int tid = threadIdx.x % T, slice = (int)(blockIdx.x / p.tiles) * S + threadIdx.x / T, tile = blockIdx.x % p.tiles;
    unsigned char *const mine = emo_smem + (threadIdx.x / T) * p.slice_bytes;
    uint32_t *const prog = reinterpret_cast<uint32_t *>(mine);
    const SliceHdr &h = *reinterpret_cast<const SliceHdr *>(mine);
    uint4 *const rec = reinterpret_cast<uint4 *>(mine + p.at_rec);
    uint32_t *const incF = reinterpret_cast<uint32_t *>(mine + p.at_inc[0]), *const incB = reinterpret_cast<uint32_t *>(mine + p.at_inc[1]);
    const bool on = slice < p.count;
    const unsigned slot_bytes = 4u * P * (unsigned)p.cols;
    const uint4 ix = on ? __ldg(p.index + slice) : make_uint4(0, 0, 0, 0);
    const uint32_t *const src = p.blob + ix.x;
    emo_slice_stage<T>(prog, src, ix.w & 0xFFFFu, tid);
    for (unsigned i = tid; i < ix.y; i += T) rec[i] = __ldg(p.rec + ix.z + i);
    __syncthreads();
    if (on) {
        emo_slice_steps<T>(mine + p.at_ops[0], src + h.dir[0].off_ops1, h.dir[0].steps, slot_bytes, 4u * P, tid);
        if (p.dirs > 1) emo_slice_steps<T>(mine + p.at_ops[1], src + h.dir[1].off_ops1, h.dir[1].steps, slot_bytes, 4u * P, tid);
    }
    emo_grid_wait_previous();            // (who wrote the levels, who read the workspace)
    emo_grid_allow_next();
    const int64_t b = (int64_t)tile * P + tid % P;
    double *const red = reinterpret_cast<double *>(emo_smem + p.at_red);
    red[threadIdx.x] = on ? emo_slice_look<P, T, true>(p, h, rec, incF, incB, b, tid) : 0.0;
    __syncthreads();
    if (on) emo_slice_sums<P, T>(h, prog, incF, incB, p.dirs, tid);
    __syncthreads();
    if (on && tid < P) {
        double e = 0.0;
        for (int k = 0; k < T / P; ++k) e += red[threadIdx.x + k * P];
        p.epart[(size_t)slice * p.nbp + b] = e;
    }
    // columns: backward first, it is the longer one
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, cw = p.cols, warps = (S * P * cw + 31) / 32;
    for (int t = warp + (p.dirs > 1 ? 0 : warps); t < 2 * warps; t += NT / 32) {
        const bool bwd = t < warps;
        const int q = (bwd ? t : t - warps) * 32 + lane, sq = q / (P * cw), r = q - sq * P * cw, pl = r / cw, col = r - pl * cw;
        const int sl = (int)(blockIdx.x / p.tiles) * S + sq;
        if (sq >= S || sl >= p.count) continue;
        unsigned char *const theirs = emo_smem + sq * p.slice_bytes;
        const emo::SliceDirHdr &hd = reinterpret_cast<const SliceHdr *>(theirs)->dir[bwd ? 1 : 0];
        if (col >= (int)hd.cols) continue;
        const unsigned base = emo_smem_addr(theirs), vals = base + (bwd ? p.at_slot[1] : p.at_slot[0]) + 4u * (unsigned)r, inc = base + (bwd ? p.at_inc[1] : p.at_inc[0]) + 4u * (unsigned)pl;
        for (unsigned j = 0; j < hd.cols; ++j) emo_slice_st(vals + j * slot_bytes, (int)j == col ? 0 : kSliceNone32);
        emo_slice_ops<int>(base + (bwd ? p.at_ops[1] : p.at_ops[0]), hd.steps, vals, inc);
        // the whole matrix is written: rows and columns that this slice has not are absent ones
        int32_t *const out = (bwd ? p.mat[1] : p.mat[0]) + (((int64_t)sl * p.nbp + (int64_t)tile * P + pl) * cw) * cw;
        const uint32_t *const ow = reinterpret_cast<const uint32_t *>(theirs) + hd.off_out;
        const unsigned outs = hd.outs, cols = hd.cols;
        for (unsigned i = 0; i < (unsigned)cw; ++i) {
            int y = kSliceNone32;
            if (i < outs) {
                const uint32_t o = ow[i];
                int v, e;
                emo_slice_ld(v, vals + (o & 0xFFFFu) * slot_bytes);
                emo_slice_ld(e, inc + (o >> 16) * (4u * P));
                y = max(v + e, kSliceNone32);
            }
            out[i * (unsigned)cw + (unsigned)col] = y;
            if (col == 0)
                for (unsigned j = cols; j < (unsigned)cw; ++j) out[i * (unsigned)cw + j] = kSliceNone32;
        }
    }
}

// 16-byte asynchronous copy
__device__ __forceinline__ void emo_slice_cp16(void *dst, const void *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}

// Matrices of one policy and direction in walking order, through a ring of D buffers in shared memory (this unit's LPP threads).
template <int LPP, int D, typename Source>
__device__ __forceinline__ void emo_slice_fetch(unsigned char *ring, int bytes, int s, int steps, int l, Source source)
{
    if (s < steps) {
        const unsigned char *const src = reinterpret_cast<const unsigned char *>(source(s));
        unsigned char *const dst = ring + (size_t)bytes * (s % D);
        for (int i = l * 16; i < bytes; i += LPP * 16) emo_slice_cp16(dst + i, src + i);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
}

// Sum of n energies, `pitch` apart, by the LPP threads of a unit in a fixed order (for thread 0).
template <int LPP>
__device__ __forceinline__ double emo_slice_energy(const double *e, int n, int64_t pitch, int l)
{
    double sum = 0.0;
    for (int k = l; k < n; k += LPP) sum += __ldcg(e + k * pitch);
    for (int o = LPP / 2; o > 0; o >>= 1) sum += __shfl_down_sync(0xFFFFFFFFu, sum, o, LPP);
    return sum;
}

// The product of a group's matrices: LPP threads per unit (policy, direction, group), a thread per column of the product, in
// registers.  x[l]: the column so far; row 0 collects the terminal nodes' maximum and enters the next matrix as the time zero, which
// column 0 has at zero and the others have not.
template <int LPP, int D, int CW>
__global__ void __launch_bounds__(32) emo_slice_group(SliceParams p)
{
    extern __shared__ __align__(128) unsigned char emo_smem[];
    constexpr int UNITS = 32 / LPP, BYTES = CW * CW * 4;
    const int sub = threadIdx.x / LPP, l = threadIdx.x % LPP, dir = blockIdx.y;
    unsigned char *const ring = emo_smem + (size_t)sub * BYTES * D;
    const int64_t unit = (int64_t)blockIdx.x * UNITS + sub, b = unit % p.nbp;
    const int g = (int)(unit / p.nbp);
    emo_grid_wait_previous();
    emo_grid_allow_next();
    const int lo = g < p.groups ? g * p.group : 0, steps = g < p.groups ? min(p.group, p.count - lo) : 0, hi = lo + steps;
    const int32_t *const mat = dir ? p.mat[1] : p.mat[0];
    auto source = [&](int s) { return mat + ((size_t)(dir == 0 ? lo + s : hi - 1 - s) * p.nbp + b) * (size_t)(CW * CW); };
    for (int s = 0; s < D - 1; ++s) emo_slice_fetch<LPP, D>(ring, BYTES, s, steps, l, source);
    if (dir == 0) {
        const double e = emo_slice_energy<LPP>(p.epart + (size_t)lo * p.nbp + b, steps, p.nbp, l);
        if (l == 0 && g < p.groups) p.gepart[(size_t)g * p.nbp + b] = e;
    }
    int x[CW], first = kSliceNone32;      // first: the maximum of row 0 so far
#pragma unroll
    for (int i = 0; i < CW; ++i) x[i] = i == l ? 0 : kSliceNone32;
    for (int s = 0; s < p.group; ++s) {
        asm volatile("cp.async.wait_group %0;" ::"n"(D - 2) : "memory");
        __syncwarp();
        emo_slice_fetch<LPP, D>(ring, BYTES, s + D - 1, steps, l, source);
        if (s < steps) {
            const int4 *const m = reinterpret_cast<const int4 *>(ring + (size_t)BYTES * (s % D));
            int y[CW];
#pragma unroll
            for (int i = 0; i < CW; ++i) {
                int best = kSliceNone32;
#pragma unroll
                for (int j = 0; j < CW / 4; ++j) {
                    const int4 r = m[i * (CW / 4) + j];
                    best = max(max(best, r.x + x[4 * j]), r.y + x[4 * j + 1]);
                    best = max(max(best, r.z + x[4 * j + 2]), r.w + x[4 * j + 3]);
                }
                y[i] = best;
            }
            first = max(first, y[0]);
            x[0] = l == 0 ? 0 : kSliceNone32;
#pragma unroll
            for (int i = 1; i < CW; ++i) x[i] = y[i];
        }
        __syncwarp();
    }
    if (g < p.groups && l < CW) {
        int32_t *const out = (dir ? p.gmat[1] : p.gmat[0]) + ((size_t)g * p.nbp + b) * (size_t)(CW * CW) + l;
        out[0] = first;
#pragma unroll
        for (int i = 1; i < CW; ++i) out[i * CW] = x[i];
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
}

// What the end of a chain leaves: makespan and energy of policy b; sums that the values' kernel adds to.
__device__ __forceinline__ void emo_slice_totals(const SliceParams &p, int64_t b, long long T, double e)
{
    if (b < p.B) {
        p.makespan[b] = T;
        p.energy[b] = e;
        if (p.slack_sum) p.slack_sum[b] = 0;
        if (p.n_critical) p.n_critical[b] = 0;
    } else if (b == p.B && b < p.nb) {
        if (p.base_T) *p.base_T = T;
        if (p.base_E) *p.base_E = e;
    }
}

// Values that enter every slice: LPP threads per unit (policy, direction, group), a thread per row of a matrix.  64-bit.
template <int LPP, int D, int CW>
__global__ void __launch_bounds__(32) emo_slice_scan(SliceParams p)
{
    extern __shared__ __align__(128) unsigned char emo_smem[];
    constexpr int UNITS = 32 / LPP;
    constexpr int cw = CW, bytes = CW * CW * 4;
    const int sub = threadIdx.x / LPP, l = threadIdx.x % LPP, dir = blockIdx.y;
    unsigned char *const ring = emo_smem + (size_t)sub * ((size_t)bytes * D + (size_t)2 * cw * 8);
    long long *const c = reinterpret_cast<long long *>(ring + (size_t)bytes * D);      // [2][cw]
    // groups in walking order, the policies of one group side by side
    const int64_t unit = (int64_t)blockIdx.x * UNITS + sub, b = unit % p.nbp;
    const int gw = (int)(unit / p.nbp);
    emo_grid_wait_previous();
    emo_grid_allow_next();
    const bool active = gw < p.groups;
    const int g = dir == 0 ? gw : p.groups - 1 - gw;
    const int lo = active ? g * p.group : 0, hi = active ? min(lo + p.group, p.count) : 0;
    // steps: the groups before this one, then its slices
    const int before = active ? gw : 0, steps = before + (hi - lo);
    const int32_t *const mat = dir ? p.mat[1] : p.mat[0], *const gmat = dir ? p.gmat[1] : p.gmat[0];
    long long *const state = dir ? p.state[1] : p.state[0];
    auto source = [&](int s) {
        if (s < before) return gmat + ((size_t)(dir == 0 ? s : p.groups - 1 - s) * p.nbp + b) * (size_t)(cw * cw);
        const int k = dir == 0 ? lo + (s - before) : hi - 1 - (s - before);
        return mat + ((size_t)k * p.nbp + b) * (size_t)(cw * cw);
    };
    for (int i = l; i < 2 * cw; i += LPP) c[i] = 0;
    for (int s = 0; s < D - 1; ++s) emo_slice_fetch<LPP, D>(ring, bytes, s, steps, l, source);
    long long T = 0;
    int cur = 0;
    // (a warp's units may have different lengths: all take the longest's steps)
    int most = steps;
    for (int o = 16; o > 0; o >>= 1) most = max(most, __shfl_xor_sync(0xFFFFFFFFu, most, o));
    for (int s = 0; s < most; ++s) {
        asm volatile("cp.async.wait_group %0;" ::"n"(D - 2) : "memory");
        __syncwarp();
        emo_slice_fetch<LPP, D>(ring, bytes, s + D - 1, steps, l, source);
        if (s < steps) {
            const long long *const from = c + cur * cw;
            long long *const to = c + (cur ^ 1) * cw;
            if (s >= before) {
                const int k = dir == 0 ? lo + (s - before) : hi - 1 - (s - before);
                long long *const st = state + ((size_t)k * p.nbp + b) * cw;
                for (int i = l; i < cw; i += LPP) st[i] = from[i];
            }
            const int *const m = reinterpret_cast<const int *>(ring + (size_t)bytes * (s % D));
            if (l < cw) {
                long long best = 0;      // (all values are times: never below zero)
                const int4 *const row = reinterpret_cast<const int4 *>(m + l * cw);
#pragma unroll
                for (int j = 0; j < cw; j += 4) {
                    const int4 a = row[j / 4];
                    const longlong2 f0 = reinterpret_cast<const longlong2 *>(from + j)[0], f1 = reinterpret_cast<const longlong2 *>(from + j)[1];
                    const long long t0 = a.x >= 0 ? f0.x + a.x : 0, t1 = a.y >= 0 ? f0.y + a.y : 0, t2 = a.z >= 0 ? f1.x + a.z : 0, t3 = a.w >= 0 ? f1.y + a.w : 0;
                    best = max(best, max(max(t0, t1), max(t2, t3)));
                }
                if (l == 0) T = max(T, best);
                to[l] = l == 0 ? 0 : best;
            }
            cur ^= 1;
        }
        __syncwarp();
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    // (the last group's unit has seen every slice or group)
    const bool total = dir == 0 && active && gw == p.groups - 1;
    if (dir == 0) {
        const double e = emo_slice_energy<LPP>(p.groups > 1 ? p.gepart + b : p.epart + b, total ? (p.groups > 1 ? p.groups : p.count) : 0, p.nbp, l);
        if (total && l == 0) emo_slice_totals(p, b, T, e);
    }
}

// The same for matrices of more than 16 columns, slices one by one: a block of 256 threads per policy and direction, four threads per
// row.  (One warp with two rows a thread took 1.5 us a slice at 40 columns.)
template <int D>
__global__ void __launch_bounds__(256) emo_slice_scan_wide(SliceParams p)
{
    extern __shared__ __align__(128) unsigned char emo_smem[];
    const int cw = p.cols, bytes = cw * cw * 4, dir = blockIdx.y, i = threadIdx.x >> 2, part = threadIdx.x & 3;
    const int64_t b = blockIdx.x;
    long long *const c = reinterpret_cast<long long *>(emo_smem + (size_t)bytes * D);      // [2][cw]
    emo_grid_wait_previous();
    emo_grid_allow_next();
    const int32_t *const mat = dir ? p.mat[1] : p.mat[0];
    long long *const state = dir ? p.state[1] : p.state[0];
    auto source = [&](int s) { return mat + ((size_t)(dir == 0 ? s : p.count - 1 - s) * p.nbp + b) * (size_t)(cw * cw); };
    for (int k = threadIdx.x; k < 2 * cw; k += 256) c[k] = 0;
    for (int s = 0; s < D - 1; ++s) emo_slice_fetch<256, D>(emo_smem, bytes, s, p.count, threadIdx.x, source);
    long long T = 0;
    int cur = 0;
    for (int s = 0; s < p.count; ++s) {
        asm volatile("cp.async.wait_group %0;" ::"n"(D - 2) : "memory");
        __syncthreads();                 // this matrix and the values; the buffer of the slice before is free
        emo_slice_fetch<256, D>(emo_smem, bytes, s + D - 1, p.count, threadIdx.x, source);
        const long long *const from = c + cur * cw;
        long long *const to = c + (cur ^ 1) * cw;
        if ((int)threadIdx.x < cw) state[((size_t)(dir == 0 ? s : p.count - 1 - s) * p.nbp + b) * cw + threadIdx.x] = from[threadIdx.x];
        long long best = 0;
        if (i < cw) {
            const int4 *const row = reinterpret_cast<const int4 *>(emo_smem + (size_t)bytes * (s % D) + (size_t)i * cw * 4);
            for (int j = part * 4; j < cw; j += 16) {
                const int4 a = row[j / 4];
                const longlong2 f0 = reinterpret_cast<const longlong2 *>(from + j)[0], f1 = reinterpret_cast<const longlong2 *>(from + j)[1];
                const long long t0 = a.x >= 0 ? f0.x + a.x : 0, t1 = a.y >= 0 ? f0.y + a.y : 0, t2 = a.z >= 0 ? f1.x + a.z : 0, t3 = a.w >= 0 ? f1.y + a.w : 0;
                best = max(best, max(max(t0, t1), max(t2, t3)));
            }
        }
        best = max(best, __shfl_xor_sync(0xFFFFFFFFu, best, 1));
        best = max(best, __shfl_xor_sync(0xFFFFFFFFu, best, 2));
        if (i < cw && part == 0) to[i] = i == 0 ? 0 : best;
        if (i == 0) T = max(T, best);
        cur ^= 1;
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    if (dir == 0 && threadIdx.x < 32) {
        const double e = emo_slice_energy<32>(p.epart + b, p.count, p.nbp, threadIdx.x);
        if (threadIdx.x == 0) emo_slice_totals(p, b, T, e);
    }
}

// The same with the steps as the program has them (16 bytes each): for blocks whose shared memory holds several slices.
template <typename V>
__device__ __forceinline__ void emo_slice_ops_packed(unsigned at, unsigned steps, unsigned vals, unsigned slot_bytes, unsigned inc)
{
    const V none = (V)kSliceNone32;
    V acc = none;
    uint4 w = emo_lds128(at);
    for (unsigned k = 0; k < steps; ++k) {
        V x0, x1;
        int s0, s1;
        emo_slice_ld(x0, vals + (w.x & 0xFFFFu) * slot_bytes);
        emo_slice_ld(x1, vals + (w.y & 0xFFFFu) * slot_bytes);
        emo_slice_ld(s0, inc + (w.x >> 16) * 4u);
        emo_slice_ld(s1, inc + (w.y >> 16) * 4u);
        const unsigned to = vals + w.z * slot_bytes, last = w.w;
        at += 16u;
        w = emo_lds128(at);              // (behind the last: a spare one)
        const V y = max(max(acc, x0 + (V)(unsigned)s0), x1 + (V)(unsigned)s1);
        emo_slice_st(to, y);
        acc = last ? none : y;
    }
}

// A graph of up to S slices, one policy per block: the three kernels' work without leaving the block, durations and running sums once.
// (400 nodes x 64 policies: 16.6 us a call against 21.5 for the three kernels, 1 013 x 64: 23.7 against 26.3.)
template <int S, int NT>
__global__ void __launch_bounds__(NT) emo_slice_whole(SliceParams p)
{
    extern __shared__ __align__(128) unsigned char emo_smem[];
    constexpr int T = NT / S;
    const int tid = threadIdx.x % T, sq = threadIdx.x / T, warp = threadIdx.x >> 5, lane = threadIdx.x & 31, cw = p.cols, count = p.count;
    const int64_t b = blockIdx.x;
    unsigned char *const mine = emo_smem + sq * p.slice_bytes;
    uint32_t *const prog = reinterpret_cast<uint32_t *>(mine);
    const SliceHdr &h = *reinterpret_cast<const SliceHdr *>(mine);
    uint4 *const rec = reinterpret_cast<uint4 *>(mine + p.at_rec);
    uint32_t *const incF = reinterpret_cast<uint32_t *>(mine + p.at_inc[0]), *const incB = reinterpret_cast<uint32_t *>(mine + p.at_inc[1]);
    const long long *const valsF = reinterpret_cast<const long long *>(mine + p.at_slot[0]), *const valsB = reinterpret_cast<const long long *>(mine + p.at_slot[1]);
    // behind the slices: energies (later the sums of the slack), makespan, states [2][S][cw], matrices [2][S][cw][cw]
    double *const red = reinterpret_cast<double *>(emo_smem + p.at_red);
    long long *const makespan = reinterpret_cast<long long *>(red + NT), *const state = makespan + 2;
    int *const mat = reinterpret_cast<int *>(state + 2 * S * cw);
    const bool on = sq < count;
    const uint4 ix = on ? __ldg(p.index + sq) : make_uint4(0, 0, 0, 0);
    emo_slice_stage<T>(prog, p.blob + ix.x, ix.w >> 16, tid);
    for (unsigned i = tid; i < ix.y; i += T) rec[i] = __ldg(p.rec + ix.z + i);
    emo_grid_wait_previous();
    emo_grid_allow_next();
    __syncthreads();
    red[threadIdx.x] = on ? emo_slice_look<1, T, true>(p, h, rec, incF, incB, b, tid) : 0.0;
    __syncthreads();
    if (on) emo_slice_sums<1, T>(h, prog, incF, incB, p.dirs, tid);
    __syncthreads();
    // matrices, a thread per slice and column; their values take the place of those below
    const int warps = (S * cw + 31) / 32;
    for (int t = warp + (p.dirs > 1 ? 0 : warps); t < 2 * warps; t += NT / 32) {
        const bool bwd = t < warps;
        const int q = (bwd ? t : t - warps) * 32 + lane, so = q / cw, col = q - so * cw;
        if (so >= count) continue;
        unsigned char *const theirs = emo_smem + so * p.slice_bytes;
        const emo::SliceDirHdr &hd = reinterpret_cast<const SliceHdr *>(theirs)->dir[bwd ? 1 : 0];
        int *const out = mat + ((bwd ? S : 0) + so) * cw * cw + col;
        const bool have = col < (int)hd.cols;
        const unsigned base = emo_smem_addr(theirs), slot_bytes = 4u * (unsigned)cw, vals = base + (bwd ? p.at_slot[1] : p.at_slot[0]) + 4u * (unsigned)col, inc = base + (bwd ? p.at_inc[1] : p.at_inc[0]);
        if (have) {
            for (unsigned j = 0; j < hd.cols; ++j) emo_slice_st(vals + j * slot_bytes, (int)j == col ? 0 : kSliceNone32);
            emo_slice_ops_packed<int>(base + 4u * hd.off_ops1, hd.steps, vals, slot_bytes, inc);
        }
        const uint32_t *const ow = reinterpret_cast<const uint32_t *>(theirs) + hd.off_out;
        for (unsigned i = 0; i < (unsigned)cw; ++i) {
            int y = kSliceNone32;
            if (have && i < hd.outs) {
                const uint32_t o = ow[i];
                int v, e;
                emo_slice_ld(v, vals + (o & 0xFFFFu) * slot_bytes);
                emo_slice_ld(e, inc + (o >> 16) * 4u);
                y = max(v + e, kSliceNone32);
            }
            out[i * (unsigned)cw] = y;
        }
    }
    __syncthreads();
    // the values that enter every slice: a warp per direction, a thread per row
    if (warp < p.dirs) {
        long long T0 = 0;
        long long *const st = state + warp * S * cw;
        for (int x = 0; x < count; ++x) {
            const int k = warp == 0 ? x : count - 1 - x, k_next = warp == 0 ? k + 1 : k - 1;
            if (x == 0)
                for (int j = lane; j < cw; j += 32) st[k * cw + j] = 0;
            __syncwarp();
            for (int i = lane; i < cw; i += 32) {
                const int *const row = mat + ((warp == 0 ? 0 : S) + k) * cw * cw + i * cw;
                long long best = 0;
                for (int j = 0; j < cw; ++j) {
                    const int a = row[j];
                    if (a >= 0) best = max(best, st[k * cw + j] + a);
                }
                if (i == 0) T0 = max(T0, best);
                if (x + 1 < count) st[k_next * cw + i] = i == 0 ? 0 : best;
            }
            __syncwarp();
        }
        if (warp == 0 && lane == 0) *makespan = T0;
    } else if (warp == 2) {
        double e = 0.0;
        for (int k = lane; k < NT; k += 32) e += red[k];
        for (int o = 16; o > 0; o >>= 1) e += __shfl_down_sync(0xFFFFFFFFu, e, o);
        if (lane == 0) {
            if (b < p.B) p.energy[b] = e;
            else if (p.base_E) *p.base_E = e;
        }
    }
    __syncthreads();
    const long long Tm = *makespan;
    if (threadIdx.x == 0) {
        if (b < p.B) p.makespan[b] = Tm;
        else if (p.base_T) *p.base_T = Tm;
    }
    if (p.dirs == 1 || b >= p.B) return;
    // every operation once, a thread per slice and direction
    if ((int)threadIdx.x < 2 * count) {
        const int so = threadIdx.x >> 1, dir = threadIdx.x & 1;
        unsigned char *const theirs = emo_smem + so * p.slice_bytes;
        const emo::SliceDirHdr &hd = reinterpret_cast<const SliceHdr *>(theirs)->dir[dir];
        const unsigned base = emo_smem_addr(theirs), vals = base + (dir ? p.at_slot[1] : p.at_slot[0]);
        for (unsigned j = 0; j < hd.cols; ++j) emo_slice_st(vals + 8u * j, state[(dir * S + so) * cw + (int)j]);
        emo_slice_ops_packed<long long>(base + 4u * hd.off_ops2, hd.steps, vals, 8u, base + (dir ? p.at_inc[1] : p.at_inc[0]));
    }
    __syncthreads();
    long long ssum = 0, ncrit = 0;
    if (on) {
        for (int i = tid; i < (int)ix.y; i += T) {
            const uint4 r = rec[i];
            const long long es = valsF[r.w & 0xFFFFu] + (long long)incF[(r.z & 0xFFFFu) - 1u];
            const long long ls = Tm - valsB[r.w >> 16] - (long long)incB[r.z >> 16];
            const long long sl = ls - es;
            const int64_t at = (int64_t)r.y * p.ldo + b;
            if (p.slack) p.slack[at] = sl;
            if (p.ES) p.ES[at] = es;
            if (p.LS) p.LS[at] = ls;
            ssum += sl;
            ncrit += sl == 0;
        }
    }
    if (p.slack_sum || p.n_critical) {
        long long *const part = reinterpret_cast<long long *>(red);      // (every thread has passed the barrier behind its last use)
        for (int o = 16; o > 0; o >>= 1) {
            ssum += __shfl_down_sync(0xFFFFFFFFu, ssum, o);
            ncrit += __shfl_down_sync(0xFFFFFFFFu, ncrit, o);
        }
        if (lane == 0) {
            part[2 * warp] = ssum;
            part[2 * warp + 1] = ncrit;
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            long long s = 0, c = 0;
            for (int k = 0; k < NT / 32; ++k) {
                s += part[2 * k];
                c += part[2 * k + 1];
            }
            if (p.slack_sum) p.slack_sum[b] = s;
            if (p.n_critical) p.n_critical[b] = (int32_t)c;
        }
    }
}

// ES, LS, slack of every node of a slice; SINGLE: the graph is one slice, so also the makespan and the energy.
template <int P, int S, int NT, bool SINGLE>
__global__ void __launch_bounds__(NT) emo_slice_values(SliceParams p)
{
    extern __shared__ __align__(128) unsigned char emo_smem[];
    constexpr int T = NT / S;
    const int tid = threadIdx.x % T, slice = (int)(blockIdx.x / p.tiles) * S + threadIdx.x / T, tile = blockIdx.x % p.tiles;
    unsigned char *const mine = emo_smem + (threadIdx.x / T) * p.slice_bytes;
    uint32_t *const prog = reinterpret_cast<uint32_t *>(mine);
    const SliceHdr &h = *reinterpret_cast<const SliceHdr *>(mine);
    uint4 *const rec = reinterpret_cast<uint4 *>(mine + p.at_rec);
    uint32_t *const incF = reinterpret_cast<uint32_t *>(mine + p.at_inc[0]), *const incB = reinterpret_cast<uint32_t *>(mine + p.at_inc[1]);
    long long *const valsF = reinterpret_cast<long long *>(mine + p.at_slot[0]), *const valsB = reinterpret_cast<long long *>(mine + p.at_slot[1]);
    double *const red = reinterpret_cast<double *>(emo_smem + p.at_red);
    long long *const makespan = reinterpret_cast<long long *>(red + NT);      // [P] (SINGLE)
    const bool on = slice < p.count;
    const uint4 ix = on ? __ldg(p.index + slice) : make_uint4(0, 0, 0, 0);
    const uint32_t *const src = p.blob + ix.x;
    emo_slice_stage<T>(prog, src, ix.w & 0xFFFFu, tid);
    for (unsigned i = tid; i < ix.y; i += T) rec[i] = __ldg(p.rec + ix.z + i);
    if (SINGLE) emo_grid_wait_previous();      // else the kernels before have waited for who wrote the levels
    __syncthreads();
    const int pl = tid % P;
    const int64_t b = (int64_t)tile * P + pl;
    double ea = 0.0;
    if (on) {
        emo_slice_steps<T>(mine + p.at_ops[0], src + h.dir[0].off_ops2, h.dir[0].steps, 8u * P, 4u * P, tid);
        if (p.dirs > 1) emo_slice_steps<T>(mine + p.at_ops[1], src + h.dir[1].off_ops2, h.dir[1].steps, 8u * P, 4u * P, tid);
        ea = emo_slice_look<P, T, SINGLE>(p, h, rec, incF, incB, b, tid);
    }
    __syncthreads();
    if (on) emo_slice_sums<P, T>(h, prog, incF, incB, p.dirs, tid);
    if (!SINGLE) emo_grid_wait_previous();
    emo_grid_allow_next();
    if (on) {
        for (int j = tid / P; j < (int)h.dir[0].cols; j += T / P) valsF[j * P + pl] = j == 0 ? 0 : p.state[0][((size_t)slice * p.nbp + b) * p.cols + j];
        if (p.dirs > 1)
            for (int j = tid / P; j < (int)h.dir[1].cols; j += T / P) valsB[j * P + pl] = j == 0 ? 0 : p.state[1][((size_t)slice * p.nbp + b) * p.cols + j];
    }
    if (SINGLE) red[threadIdx.x] = ea;
    __syncthreads();
    // the operations: a thread per slice, direction and policy
    if ((int)threadIdx.x < S * P * p.dirs) {
        const int sq = threadIdx.x / (P * p.dirs), r = threadIdx.x - sq * P * p.dirs, po = r % P, sl = (int)(blockIdx.x / p.tiles) * S + sq;
        const bool fwd = r < P;
        if (sl < p.count) {
            unsigned char *const theirs = emo_smem + sq * p.slice_bytes;
            const SliceHdr &ho = *reinterpret_cast<const SliceHdr *>(theirs);
            const unsigned base = emo_smem_addr(theirs);
            emo_slice_ops<long long>(base + (fwd ? p.at_ops[0] : p.at_ops[1]), fwd ? ho.dir[0].steps : ho.dir[1].steps, base + (fwd ? p.at_slot[0] : p.at_slot[1]) + 8u * (unsigned)po,
                                     base + (fwd ? p.at_inc[0] : p.at_inc[1]) + 4u * (unsigned)po);
            if (SINGLE && fwd) {
                const long long Tm = valsF[ho.dir[0].term * P + po];
                double e = 0.0;
                for (int k = 0; k < NT / P; ++k) e += red[k * P + po];
                makespan[po] = Tm;
                const int64_t bo = (int64_t)tile * P + po;
                if (bo < p.B) {
                    p.makespan[bo] = Tm;
                    p.energy[bo] = e;
                } else if (bo == p.B && bo < p.nb) {
                    if (p.base_T) *p.base_T = Tm;
                    if (p.base_E) *p.base_E = e;
                }
            }
        }
    }
    if (p.dirs == 1) return;
    __syncthreads();
    const bool real = on && b < p.B;
    const long long Tm = SINGLE ? makespan[pl] : (real ? p.makespan[b] : 0);
    long long ssum = 0;
    int ncrit = 0;
    if (real) {
        for (int i = tid / P; i < (int)ix.y; i += T / P) {
            const uint4 r = rec[i];
            const long long es = valsF[(r.w & 0xFFFFu) * P + pl] + (long long)incF[((r.z & 0xFFFFu) - 1u) * P + pl];
            const long long ls = Tm - valsB[(r.w >> 16) * P + pl] - (long long)incB[(r.z >> 16) * P + pl];
            const long long sl = ls - es;
            const int64_t at = (int64_t)r.y * p.ldo + b;
            if (p.slack) p.slack[at] = sl;
            if (p.ES) p.ES[at] = es;
            if (p.LS) p.LS[at] = ls;
            ssum += sl;
            ncrit += sl == 0;
        }
    }
    if (p.slack_sum || p.n_critical) {
        // a thread per slice and policy adds its slice's parts
        long long *const part = reinterpret_cast<long long *>(red);
        __syncthreads();
        part[threadIdx.x] = ssum;
        __syncthreads();
        long long s = 0, c = 0;
        if (tid < P)
            for (int k = 0; k < T / P; ++k) s += part[threadIdx.x + k * P];
        __syncthreads();
        part[threadIdx.x] = ncrit;
        __syncthreads();
        if (tid < P && real) {
            for (int k = 0; k < T / P; ++k) c += part[threadIdx.x + k * P];
            if (SINGLE) {
                if (p.slack_sum) p.slack_sum[b] = s;
                if (p.n_critical) p.n_critical[b] = (int32_t)c;
            } else {
                // (whole numbers: the order of the slices does not matter)
                if (p.slack_sum) atomicAdd(reinterpret_cast<unsigned long long *>(p.slack_sum + b), (unsigned long long)s);
                if (p.n_critical) atomicAdd(p.n_critical + b, (int32_t)c);
            }
        }
    }
}
