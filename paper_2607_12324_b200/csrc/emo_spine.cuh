// The spine kernels (sm_100a): emo_spine_fwd and emo_spine_bwd walk the spine program of emo_flow.h.
// Included only by emo_lib.cu.
//
// A block holds a tile of ptile = 32 * groups policies.  The recurrence of Eq. 1 runs through the spine warps alone:
// per segment the maximum of two value slots plus the segment's sum, in the spine's own program order, so no value is
// ever waited for inside a stage and an operation has neither a branch nor a predicate.  The operations come in bundles
// of NB that do not depend on each other; a spine warp works on a whole bundle at once, 32 / NB of its threads on every
// operation, VS policies per thread.  Everything else is done by other warps around it:
//   look-up workers   levels, table look-ups, the sums per segment, the energy (forward); VW policies per thread
//   forward, pushers  completion offsets that the backward pass cannot derive, from the buffer of sums to the restore list
//   backward, walkers the lanes' completion offsets, ahead of the spine (a subtraction per segment, or a restored word);
//                     NB lanes at a time, as the spine does with operations
//   backward, stores  behind the spine: the slack of every member (one number per segment) and the tails that nodes of much
//                     earlier stages read (folded into a slot of the reader with a maximum); VW policies per thread
//   two producers     one brings the workers' part of a stage and the level rows of the tile, one the spine's part, each
//                     into a ring of its own, so that a stage's tables are released as soon as its sums are taken
// A stage's look-up entries are cut into chunks at segment boundaries; a chunk is the workers' unit of work and worker k
// takes every n-th one, which keeps the order of the energy sums fixed.
//
// What bounds it: with many policies per SM the shared-memory pipe and the issue slots (a look-up is three shared loads
// of four bytes per node and policy, forward), backward the stores of the slack matrix; with one policy group per SM the
// spine's operations.  What one warp alone pays, in cycles: a dependent shared load 29 (a predicated one 33 even when it
// is off), a store or maximum 5 .. 11 (also when off), a 128-bit broadcast load 2, a branch on a freshly loaded word 100 and
// more.  Hence several policies per thread (the records, addresses and level words of an entry are loaded once for 64 or
// 128 policies), operations without predicates, a bundle per instruction, loops over flat lists instead of segments.
//
// Inside a sub-tile of 32 * VW policies the slots, sums and restore rows hold policy VW * l + v at word 32 * v + l: a
// worker thread l has consecutive policies (one load for their level bytes, one store for their results) and the 32
// threads of a warp still meet in 32 different banks.
//
// Every wait is bounded (wait_cycles); a wait that runs out sets the block's abort word, which ends every
// other wait of the block early, and EMO_E_TIMEOUT goes to *status.  A barrier's parity tells two phases
// apart, so a warp may wait for a phase only when the one before it has completed: a worker must not skip more stages
// than a ring of sums has buffers (the launch gives a sub-tile at most chunks * nacc workers).
#pragma once
#include "emo_flow.cuh"

constexpr int kSpRing = 8;               // most buffers of a ring
constexpr int kSpChunks = 16;            // most chunks of a stage and kind (look-up, storing)
constexpr int kSpRowRing = 4;            // stages whose row numbers are on their way or in use

struct SpineParams {
    const unsigned char *blobW;          // [stages][w_bytes] the workers' part: chunk table (4 * 2 * kSpChunks bytes), position words, (backward) member
                                         // records, bits of the segments' first entries, table rows
    const unsigned char *blobS;          // [stages][s_bytes] the spine's part: header, (forward) terminal nodes, operations, records of the pushers or the
                                         // completion walk
    const uint32_t *rows;                // [stages][nlook] policy row of every look-up entry (kNone: none)
    const uint32_t *push_base;           // [stages + 1] first restore row of every stage
    unsigned w_bytes, s_bytes, off_pos, off_tab, tab_row, off_ops;
    unsigned off_mem, off_first, off_rec;      // backward: members, a bit per entry (first of its segment); forward: records of the pushers, backward: of the completion walk
    int nlook;                           // look-up entries that a stage has room for (entries behind them have none)
    int chunks, chunks_post;             // per stage: look-up chunks; backward: chunks of the storing workers
    int stages, lanes, Lp, L;
    int groups, ptile;
    int workers, posts;                  // look-up warps; backward: storing warps (both multiples of the tile's sub-tiles of 32 * VW); forward: pushers
    int nw, ns, nacc;                    // buffers: workers' part, spine's part, sums
    unsigned wbuf_bytes, sbuf_bytes, acc_bytes, slot_bytes;      // one buffer each; slots of the whole tile
    unsigned off_lvl, off_rst;           // inside a workers' / spine's buffer
    unsigned off_bar, off_rows, off_w0, off_s0, off_acc0;        // inside the block's shared memory (the slots come first)
    unsigned rowbuf_bytes;               // one stage's row numbers
    unsigned zero_word;                  // word of a buffer of sums that stays zero
    unsigned comp_off;                   // backward: from a segment's sum (later its qin) to its completion offset, in units of 128 bytes per group
    int c_slot0;                         // backward: first slot of the lanes' completion offsets
    int want_base;
    int64_t B;
    const uint8_t *lvl;
    int64_t ldb;
    uint32_t *restore;                   // [tiles][restore_rows][ptile]
    int64_t restore_rows, pushes;        // restore_rows = pushes + lanes
    int64_t *makespan;
    double *energy;
    int64_t *base_T;
    double *base_E;
    int64_t *ES, *LS, *slack;
    int64_t ldo;
    int vec_out;                         // outputs may be stored VW policies at a time (pitch and pointers aligned)
    int64_t *slack_sum;
    int32_t *n_critical;
    int32_t *status;
    long long wait_cycles;
    int stall_stage;                     // test hook: the producers stop before this stage (-1: off)
    long long *prof;
};

// ---- waits ------------------------------------------------------------------------------------------------
// try_wait with a time to stay suspended: a waiting warp takes no issue slots.  (Polling with naps in between took 40 % of
// all executed instructions and, in a function of its own, pushed the working warps' loops out of the instruction cache.)
__device__ __forceinline__ bool emo_mbar_suspend(unsigned bar, unsigned parity)
{
    unsigned ok;
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(ok) : "r"(bar), "r"(parity), "r"(20000u) : "memory");
    return ok != 0;
}
__device__ __forceinline__ bool emo_spine_wait(unsigned bar, unsigned parity, volatile int *abort_word, long long limit)
{
    if (emo_mbar_suspend(bar, parity)) return true;
    const long long t0 = clock64();
    while (!emo_mbar_suspend(bar, parity))
        if (*abort_word || clock64() - t0 > limit) return false;
    return true;
}

// ---- shared-memory accesses of V policies -----------------------------------------------------------------
template <int V>
struct EmoVec {
    unsigned v[V];
};
template <int V>
__device__ __forceinline__ EmoVec<V> emo_ldv(unsigned a)
{
    EmoVec<V> r;
    if constexpr (V == 1) asm volatile("ld.shared.u32 %0, [%1];" : "=r"(r.v[0]) : "r"(a));
    if constexpr (V == 2) asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(r.v[0]), "=r"(r.v[1]) : "r"(a));
    if constexpr (V == 4)
        asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(r.v[0]), "=r"(r.v[1]), "=r"(r.v[2]), "=r"(r.v[3]) : "r"(a));
    return r;
}
// the words at a where `take` is set, else `r` as it was (no access, no branch)
template <int V>
__device__ __forceinline__ void emo_ldv_if(EmoVec<V> &r, unsigned a, unsigned take)
{
    if constexpr (V == 1) asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %2, 0;\n\t@p ld.shared.u32 %0, [%1];\n\t}" : "+r"(r.v[0]) : "r"(a), "r"(take));
    if constexpr (V == 2)
        asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %3, 0;\n\t@p ld.shared.v2.u32 {%0, %1}, [%2];\n\t}" : "+r"(r.v[0]), "+r"(r.v[1]) : "r"(a), "r"(take));
    if constexpr (V == 4)
        asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %5, 0;\n\t@p ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];\n\t}"
                     : "+r"(r.v[0]), "+r"(r.v[1]), "+r"(r.v[2]), "+r"(r.v[3]) : "r"(a), "r"(take));
}
template <int V>
__device__ __forceinline__ void emo_stv(unsigned a, const EmoVec<V> &r)
{
    if constexpr (V == 1) asm volatile("st.shared.u32 [%0], %1;" ::"r"(a), "r"(r.v[0]) : "memory");
    if constexpr (V == 2) asm volatile("st.shared.v2.u32 [%0], {%1, %2};" ::"r"(a), "r"(r.v[0]), "r"(r.v[1]) : "memory");
    if constexpr (V == 4) asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(a), "r"(r.v[0]), "r"(r.v[1]), "r"(r.v[2]), "r"(r.v[3]) : "memory");
}
template <int V>
__device__ __forceinline__ void emo_stv_if(unsigned a, const EmoVec<V> &r, unsigned ok)
{
    if constexpr (V == 1) asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %2, 0;\n\t@p st.shared.u32 [%0], %1;\n\t}" ::"r"(a), "r"(r.v[0]), "r"(ok) : "memory");
    if constexpr (V == 2)
        asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %3, 0;\n\t@p st.shared.v2.u32 [%0], {%1, %2};\n\t}" ::"r"(a), "r"(r.v[0]), "r"(r.v[1]), "r"(ok) : "memory");
    if constexpr (V == 4)
        asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %5, 0;\n\t@p st.shared.v4.u32 [%0], {%1, %2, %3, %4};\n\t}" ::"r"(a), "r"(r.v[0]), "r"(r.v[1]),
                     "r"(r.v[2]), "r"(r.v[3]), "r"(ok) : "memory");
}
// V words of a restore row under a predicate: base + row * pitch
template <int V>
__device__ __forceinline__ void emo_stg_row_if(uint32_t *base, unsigned row, unsigned pitch_bytes, const EmoVec<V> &r, unsigned ok)
{
    if constexpr (V == 1)
        asm volatile("{\n\t.reg .pred p;\n\t.reg .u64 a;\n\tsetp.ne.u32 p, %4, 0;\n\tmad.wide.u32 a, %1, %2, %0;\n\t@p st.global.u32 [a], %3;\n\t}" ::"l"(base),
                     "r"(row), "r"(pitch_bytes), "r"(r.v[0]), "r"(ok) : "memory");
    if constexpr (V == 2)
        asm volatile("{\n\t.reg .pred p;\n\t.reg .u64 a;\n\tsetp.ne.u32 p, %5, 0;\n\tmad.wide.u32 a, %1, %2, %0;\n\t@p st.global.v2.u32 [a], {%3, %4};\n\t}" ::"l"(base),
                     "r"(row), "r"(pitch_bytes), "r"(r.v[0]), "r"(r.v[1]), "r"(ok) : "memory");
    if constexpr (V == 4)
        asm volatile("{\n\t.reg .pred p;\n\t.reg .u64 a;\n\tsetp.ne.u32 p, %7, 0;\n\tmad.wide.u32 a, %1, %2, %0;\n\t@p st.global.v4.u32 [a], {%3, %4, %5, %6};\n\t}" ::"l"(base),
                     "r"(row), "r"(pitch_bytes), "r"(r.v[0]), "r"(r.v[1]), "r"(r.v[2]), "r"(r.v[3]), "r"(ok) : "memory");
}
// V 64-bit outputs of one node at once (under a predicate)
template <int V>
__device__ __forceinline__ void emo_stg_out_if(long long *base, unsigned row, unsigned pitch_bytes, const long long (&x)[V], unsigned ok)
{
    if constexpr (V == 1)
        asm volatile("{\n\t.reg .pred p;\n\t.reg .u64 a;\n\tsetp.ne.u32 p, %4, 0;\n\tmad.wide.u32 a, %1, %2, %0;\n\t@p st.global.b64 [a], %3;\n\t}" ::"l"(base), "r"(row),
                     "r"(pitch_bytes), "l"(x[0]), "r"(ok) : "memory");
    if constexpr (V == 2)
        asm volatile("{\n\t.reg .pred p;\n\t.reg .u64 a;\n\tsetp.ne.u32 p, %5, 0;\n\tmad.wide.u32 a, %1, %2, %0;\n\t@p st.global.v2.b64 [a], {%3, %4};\n\t}" ::"l"(base), "r"(row),
                     "r"(pitch_bytes), "l"(x[0]), "l"(x[1]), "r"(ok) : "memory");
    if constexpr (V == 4)
        asm volatile("{\n\t.reg .pred p;\n\t.reg .u64 a;\n\tsetp.ne.u32 p, %7, 0;\n\tmad.wide.u32 a, %1, %2, %0;\n\t@p st.global.v4.b64 [a], {%3, %4, %5, %6};\n\t}" ::"l"(base), "r"(row),
                     "r"(pitch_bytes), "l"(x[0]), "l"(x[1]), "l"(x[2]), "l"(x[3]), "r"(ok) : "memory");
}
// 16-byte asynchronous copy of a piece of matrix row `row` (kNone: no copy)
__device__ __forceinline__ void emo_cp_async16_row(unsigned dst, const uint8_t *base, unsigned row, unsigned pitch)
{
    asm volatile("{\n\t.reg .pred p;\n\t.reg .u64 a;\n\tsetp.ne.u32 p, %2, 0xFFFFFFFF;\n\tmad.wide.u32 a, %2, %3, %1;\n\t@p cp.async.cg.shared.global [%0], [a], 16;\n\t}" ::"r"(dst),
                 "l"(base), "r"(row), "r"(pitch) : "memory");
}
#define EMO_SCLK() (p.prof ? clock64() : 0LL)

// Position in a ring of n buffers and the parity of its current use, kept by steps (no division).
struct SpineRing {
    int idx = 0, par = 0, n = 1;
    __device__ __forceinline__ void next()
    {
        if (++idx == n) {
            idx = 0;
            par ^= 1;
        }
    }
};
enum SpineBar { kBarWFull, kBarWEmpty, kBarSFull, kBarSEmpty, kBarSums, kBarComp, kBarSpine, kBarPost, kBarRows, kBarKinds };
constexpr unsigned kSpBarBytes = kBarKinds * kSpRing * 8 + 16;      // the barriers, then the abort word and a word that is never set
__device__ __forceinline__ unsigned emo_spine_bar(unsigned bar0, SpineBar kind, int i) { return bar0 + (unsigned)(((int)kind * kSpRing + i) * 8); }

// Which warp does what: spines, (backward) completion walkers, look-up workers, storing workers (forward: pushers), two producers.
struct SpineRole {
    bool spine, comp, look, post, prod;
    int idx;                             // index among the warps of its role
};
__device__ __forceinline__ SpineRole emo_spine_role(const SpineParams &p, int warp, int spines, bool bwd)
{
    SpineRole r;
    const int w0 = spines, w1 = w0 + (bwd ? spines : 0), w2 = w1 + p.workers, w3 = w2 + p.posts;
    r.spine = warp < w0;
    r.comp = warp >= w0 && warp < w1;
    r.look = warp >= w1 && warp < w2;
    r.post = warp >= w2 && warp < w3;
    r.prod = warp >= w3;
    r.idx = r.spine ? warp : (r.comp ? warp - w0 : (r.look ? warp - w1 : (r.post ? warp - w2 : warp - w3)));
    return r;
}
__device__ __forceinline__ void emo_spine_init(const SpineParams &p, unsigned char *smem, unsigned bar0, int spines, int subs, bool bwd)
{
    unsigned *w = reinterpret_cast<unsigned *>(smem);
    for (unsigned i = threadIdx.x; i < p.slot_bytes / 4u; i += blockDim.x) w[i] = 0u;
    for (int a = 0; a < p.nacc; ++a)
        for (int i = threadIdx.x; i < p.ptile; i += blockDim.x)
            w[(p.off_acc0 + (unsigned)a * p.acc_bytes) / 4u + p.zero_word * (unsigned)p.ptile + (unsigned)i] = 0u;
    if (threadIdx.x == 0) {
        const unsigned jobs = (unsigned)(p.chunks * subs), jobs_post = bwd ? (unsigned)(p.chunks_post * subs) : 0u;
        for (int i = 0; i < kSpRing; ++i) {
            emo_mbar_init(emo_spine_bar(bar0, kBarWFull, i), 1 + 32);
            emo_mbar_init(emo_spine_bar(bar0, kBarWEmpty, i), jobs + jobs_post);
            emo_mbar_init(emo_spine_bar(bar0, kBarSFull, i), 1);
            emo_mbar_init(emo_spine_bar(bar0, kBarSEmpty, i), (unsigned)(bwd ? 2 * spines : spines + p.posts));
            emo_mbar_init(emo_spine_bar(bar0, kBarRows, i), 1);
            emo_mbar_init(emo_spine_bar(bar0, kBarSums, i), jobs);
            emo_mbar_init(emo_spine_bar(bar0, kBarComp, i), (unsigned)spines);
            emo_mbar_init(emo_spine_bar(bar0, kBarSpine, i), (unsigned)spines);
            emo_mbar_init(emo_spine_bar(bar0, kBarPost, i), bwd ? jobs_post : (unsigned)max(p.posts, 1));
        }
        volatile int *abort_word = reinterpret_cast<volatile int *>(smem + p.off_bar + kBarKinds * kSpRing * 8);
        abort_word[0] = 0;
        abort_word[1] = 0;      // never set: the drain after a failure waits its full time
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    __syncthreads();
}

// The producer warps.  Warp 0 brings the workers' part of a stage (one bulk copy) and the tile's bytes of every level row
// it reads, as 16-byte cp.async pieces (one bulk copy per row was 65 cycles of issue each: 4 100 cycles per stage of 64
// rows, twice what everything else of a forward stage takes); the row numbers come through a ring of their own, three
// stages ahead, and are read where they are used: the loop stays small (held in registers, unrolled, they made 17 KB of code
// that pushed the other warps' loops out of the instruction cache at every stage).  Warp 1 brings the spine's part and,
// backward, the stage's rows of the restore list.  Stages are issued in walking order (backward: last first).
template <bool BWD>
__device__ __forceinline__ void emo_spine_produce(const SpineParams &p, unsigned smem0, unsigned bar0, volatile int *abort_word, int lane, int which)
{
    const int stages = p.stages, nbuf = which == 0 ? p.nw : p.ns;
    const SpineBar full_k = which == 0 ? kBarWFull : kBarSFull, empty_k = which == 0 ? kBarWEmpty : kBarSEmpty;
    const int64_t b0 = (int64_t)blockIdx.x * p.ptile;
    const int64_t left = p.lvl ? p.ldb - b0 : 0;
    const unsigned lvl_bytes = left > 0 ? (unsigned)min((int64_t)p.ptile, left) : 0u, P = (unsigned)p.ptile, ldb = (unsigned)p.ldb;
    // pieces of a full row (2 .. 16) by lanes, rounded up to a power of two (tiles of 96 and 192 policies leave a quarter of the
    // lanes without one; dividing the lanes by the pieces made the forward pass 1.5 % slower); this lane's piece, and its row among
    // those of one instruction
    const int pshift = 32 - __clz((p.ptile >> 4) - 1);
    const unsigned pc16 = ((unsigned)lane & ((1u << pshift) - 1u)) * 16u, sub_row = (unsigned)lane >> pshift, step = 32u >> pshift;
    // rows of this lane: none where its piece lies beyond the tile or the matrix
    const unsigned n_rows = pc16 < lvl_bytes ? (unsigned)p.nlook : 0u;
    const uint8_t *const lvl0 = p.lvl + b0 + pc16;
    const unsigned row_bytes = (unsigned)p.nlook * 4u;
    int issued = 0, rows_issued = 0;
    bool gave_up = false;
    long long t_wait = 0, t_issue = 0;
    const long long t_begin = EMO_SCLK();
    SpineRing ring, rrow;
    ring.n = nbuf;
    rrow.n = kSpRowRing;
    auto fetch_rows = [&]() {            // the next stage's row numbers
        if (which == 0 && rows_issued < stages && lane == 0) {
            const int st = BWD ? stages - 1 - rows_issued : rows_issued, k = rows_issued % kSpRowRing;
            emo_mbar_expect_tx(emo_spine_bar(bar0, kBarRows, k), row_bytes);
            emo_bulk_g2s(smem0 + p.off_rows + (unsigned)k * p.rowbuf_bytes, p.rows + (size_t)st * p.nlook, row_bytes, emo_spine_bar(bar0, kBarRows, k));
        }
        ++rows_issued;
    };
    for (int k = 0; k < kSpRowRing - 1; ++k) fetch_rows();
    for (int c = 0; c < stages; ++c) {
        const int st = BWD ? stages - 1 - c : c;
        const int s = ring.idx;
        unsigned rst_rows = 0, rst_first = 0;
        if (BWD && which == 1) {
            rst_first = __ldg(p.push_base + st);
            rst_rows = __ldg(p.push_base + st + 1) - rst_first;
        }
        if (BWD && which == 0 && c == nbuf) emo_grid_wait_previous();      // (no wait for other warps runs while these may not)
        const long long tw0 = EMO_SCLK();
        bool ok = c < nbuf || emo_spine_wait(emo_spine_bar(bar0, empty_k, s), ring.par ^ 1, abort_word, p.wait_cycles);
        ok = ok && (which != 0 || emo_spine_wait(emo_spine_bar(bar0, kBarRows, rrow.idx), rrow.par, abort_word, p.wait_cycles));
        if (!ok) {
            if (lane == 0) {
                *abort_word = 1;
                if (p.status) atomicMin(p.status, -8);
            }
            gave_up = true;
            break;
        }
        if (__any_sync(0xFFFFFFFFu, *abort_word != 0) || c == p.stall_stage) { gave_up = true; break; }
        const long long tw1 = EMO_SCLK();
        t_wait += tw1 - tw0;
        issued = c + 1;
        const unsigned full = emo_spine_bar(bar0, full_k, s);
        if (which == 1) {
            if (lane == 0) {
                const unsigned dst = smem0 + p.off_s0 + (unsigned)s * p.sbuf_bytes, rst_bytes = rst_rows * P * 4u;
                emo_mbar_expect_tx(full, p.s_bytes + rst_bytes);
                if (BWD && c == 0) asm volatile("fence.proxy.async;" ::: "memory");      // the restore list was written by ordinary stores
                emo_bulk_g2s(dst, p.blobS + (size_t)st * p.s_bytes, p.s_bytes, full);
                if (BWD && rst_bytes)
                    emo_bulk_g2s(dst + p.off_rst, p.restore + ((size_t)blockIdx.x * p.restore_rows + rst_first) * P, rst_bytes, full);
            }
        } else {
            const unsigned dst = smem0 + p.off_w0 + (unsigned)s * p.wbuf_bytes;
            if (lane == 0) {
                emo_mbar_expect_tx(full, p.w_bytes);
                emo_bulk_g2s(dst, p.blobW + (size_t)st * p.w_bytes, p.w_bytes, full);
            }
            const unsigned rows_a = smem0 + p.off_rows + (unsigned)rrow.idx * p.rowbuf_bytes, dl = dst + p.off_lvl + pc16;
#pragma unroll 1
            for (unsigned e0 = sub_row; e0 < n_rows; e0 += 4u * step) {
                unsigned row[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) row[j] = emo_lds_u32(rows_a + (e0 + step * j) * 4u);          // (past the last: read, not used)
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const unsigned e = e0 + step * (unsigned)j;
                    emo_cp_async16_row(dl + e * P, lvl0, e < n_rows ? row[j] : emo::kNone, ldb);
                }
            }
            __syncwarp();
            emo_cp_async_arrive(full);
            fetch_rows();                // into the buffer read one stage ago
            rrow.next();
        }
        t_issue += EMO_SCLK() - tw1;
        ring.next();
    }
    if (p.prof && lane == 0 && blockIdx.x < 512) {
        long long *pr = p.prof + ((size_t)blockIdx.x * 32 + (threadIdx.x >> 5)) * 8;
        pr[0] = t_wait;
        pr[1] = t_issue;
        pr[2] = EMO_SCLK() - t_begin;
    }
    // Do not leave the block while copies into its shared memory may still be in flight: other warps may have given up, also after
    // the last stage was issued.  The copies land whatever the other warps do, so the limit here is the caller's or 10 ms.
    const long long drain = max(p.wait_cycles, 20000000LL);
    for (int c = max(0, issued - nbuf); c < issued; ++c)
        (void)emo_spine_wait(emo_spine_bar(bar0, full_k, c % nbuf), (c / nbuf) & 1, abort_word + 1, drain);
    if (which == 0)
        for (int c = issued; c < min(rows_issued, stages); ++c)
            (void)emo_spine_wait(emo_spine_bar(bar0, kBarRows, c % kSpRowRing), (c / kSpRowRing) & 1, abort_word + 1, drain);
}

// The level bytes of an entry for this thread's V consecutive policies, as table addresses: one load, then one dp4a per
// policy (byte * element size + row address).  keep, set: level mask, and the virtual all-max column's byte.
template <int V>
struct EmoLevels {
    unsigned a, keep, set;
    __device__ __forceinline__ void init(const SpineParams &p, int sub, int lane, int base_col)
    {
        const unsigned lmask = (unsigned)p.Lp - 1u, top = (unsigned)(p.L - 1);
        const int col = sub * 32 * V + lane * V;
        a = (unsigned)col;
        keep = set = 0;
#pragma unroll
        for (int v = 0; v < V; ++v) {
            const bool base = base_col == col + v;
            keep |= (base ? 0u : lmask) << (8 * v);
            set |= (base ? top : 0u) << (8 * v);
        }
    }
    __device__ __forceinline__ unsigned load(unsigned row) const
    {
        const unsigned w = V == 4 ? emo_lds_u32(row + a) : (V == 2 ? emo_lds_u16(row + a) : emo_lds_u8(row + a));
        return (w & keep) | set;
    }
    template <unsigned ELEM>
    __device__ __forceinline__ unsigned addr(unsigned w, int v, unsigned tab) const
    {
        return V > 1 ? __dp4a(w, ELEM << (8 * v), tab) : w * ELEM + tab;
    }
};
// policy of a sub-tile's word (see the head of this file)
template <int V>
__device__ __forceinline__ int emo_spine_policy(int word)
{
    const int sub = word / (32 * V), r = word - sub * 32 * V;
    return sub * 32 * V + (r & 31) * V + (r >> 5);
}

// The sums of one chunk: entries e0 .. e0 + n - 1 of the stage (n a multiple of four), two or four at a time so that their
// look-ups overlap, the next ones' level words fetched ahead; the running sum restarts where a segment begins and is stored
// where one ends.  Padding entries have all-zero tables and store nothing.  acc_t: this thread's first word of the sums.
template <int V, bool ENERGY>
__device__ __forceinline__ void emo_spine_sums(const SpineParams &p, const EmoLevels<V> &lev, unsigned wbuf, unsigned acc_t, unsigned e0, unsigned n,
                                               double (&ea)[V])
{
    constexpr int U = V == 4 ? 2 : 4;
    const unsigned tab_row = p.tab_row, P = (unsigned)p.ptile, P4 = P * 4u;
    unsigned pos_a = wbuf + p.off_pos + e0 * 4u, lvl_a = wbuf + p.off_lvl + e0 * P, tab_a = wbuf + p.off_tab + e0 * tab_row;
    unsigned run[V], wn[U];
#pragma unroll
    for (int v = 0; v < V; ++v) run[v] = 0;
    EmoVec<U> pn = emo_ldv<U>(pos_a);
#pragma unroll
    for (int i = 0; i < U; ++i) wn[i] = lev.load(lvl_a + (unsigned)i * P);
    for (unsigned j0 = 0; j0 < n; j0 += U) {
        const EmoVec<U> pw = pn;
        unsigned w[U], d[U][V];
        double e[U][V];
#pragma unroll
        for (int i = 0; i < U; ++i) w[i] = wn[i];
        pos_a += 4u * U;
        lvl_a += P * U;
#pragma unroll
        for (int i = 0; i < U; ++i)
#pragma unroll
            for (int v = 0; v < V; ++v) {
                const unsigned ta = lev.template addr<ENERGY ? 12u : 4u>(w[i], v, tab_a + (unsigned)i * tab_row);
                d[i][v] = emo_lds_u32(ta);
                if (ENERGY) e[i][v] = __hiloint2double((int)emo_lds_u32(ta + 4u), (int)emo_lds_u32(ta + 8u));
            }
        pn = emo_ldv<U>(pos_a);          // (past the last entry: read, not used)
#pragma unroll
        for (int i = 0; i < U; ++i) wn[i] = lev.load(lvl_a + (unsigned)i * P);
#pragma unroll
        for (int i = 0; i < U; ++i) {
            const unsigned at = acc_t + (pw.v[i] >> 16) * P4;
#pragma unroll
            for (int v = 0; v < V; ++v) {
                run[v] = ((pw.v[i] & emo::kSpPos_First) ? 0u : run[v]) + d[i][v];
                EmoVec<1> r;
                r.v[0] = run[v];
                emo_stv_if<1>(at + 128u * v, r, pw.v[i] & emo::kSpPos_Last);
                if (ENERGY) ea[v] += e[i][v];
            }
        }
        tab_a += tab_row * U;
    }
}

// The look-up workers: every n-th chunk of all stages, nacc stages ahead of whoever empties a buffer of sums (`freed`).
template <int V, bool ENERGY>
__device__ __forceinline__ bool emo_spine_look(const SpineParams &p, unsigned smem0, unsigned bar0, volatile int *abort_word, int lane, int idx, int subs, int base_col,
                                               SpineBar freed, double (&ea)[V])
{
    const int sub = idx % subs, n = p.workers / subs;
    EmoLevels<V> lev;
    lev.init(p, sub, lane, base_col);
    const unsigned col = (unsigned)(sub * 32 * V + lane) * 4u;
    long long t_full = 0, t_acc = 0;
    SpineRing rw, ra;
    rw.n = p.nw;
    ra.n = p.nacc;
    bool ok = true;
    const long long t_begin = EMO_SCLK();
    for (int c = 0, chunk = idx / subs;; chunk += n) {
        for (; chunk >= p.chunks; chunk -= p.chunks, ++c) {
            rw.next();
            ra.next();
        }
        if (c >= p.stages) break;
        const long long tw0 = EMO_SCLK();
        ok = emo_spine_wait(emo_spine_bar(bar0, kBarWFull, rw.idx), rw.par, abort_word, p.wait_cycles);
        const long long tw1 = EMO_SCLK();
        ok = ok && (c < p.nacc || emo_spine_wait(emo_spine_bar(bar0, freed, ra.idx), ra.par ^ 1, abort_word, p.wait_cycles));
        if (!ok) break;
        t_full += tw1 - tw0;
        t_acc += EMO_SCLK() - tw1;
        const unsigned wbuf = smem0 + p.off_w0 + (unsigned)rw.idx * p.wbuf_bytes;
        const unsigned ck = emo_uniform(emo_lds_u32(wbuf + 4u * (unsigned)chunk));
        emo_spine_sums<V, ENERGY>(p, lev, wbuf, smem0 + p.off_acc0 + (unsigned)ra.idx * p.acc_bytes + col, ck & 0xFFFFu, ck >> 16, ea);
        __syncwarp();
        if (lane == 0) {
            emo_mbar_arrive(emo_spine_bar(bar0, kBarSums, ra.idx));
            emo_mbar_arrive(emo_spine_bar(bar0, kBarWEmpty, rw.idx));
        }
    }
    if (p.prof && lane == 0 && blockIdx.x < 512) {
        long long *pr = p.prof + ((size_t)blockIdx.x * 32 + (threadIdx.x >> 5)) * 8;
        pr[0] = t_full;
        pr[1] = t_acc;
        pr[2] = EMO_SCLK() - t_begin;
    }
    return ok;
}

// The spine's operations of one stage, a bundle of NB at a time: this thread's operation (op_a: its first one) is
//   value = max(floor_sub(x0, d0), floor_sub(x1, d1)) + sum
// for VS policies.  All operands of a bundle are loaded before any result is stored.  The value goes to the lane's slot, to a
// published slot and to the segment's word (backward: there the maximum, qin, without the sum; and a slot that collected
// folded tails is cleared).  Absent operands and outputs name slots that stay zero / that nobody reads; the next bundle's
// words are fetched beside the operands.  (Measured on one warp, bundles of two, cycles per bundle: with all 32 threads on one
// operation after the other 114, with half a warp on each 75 and half the instructions; taking the bundle before's results
// from registers instead of slots did not pay, 120: the pipes are then full, a shared store alone takes 4.5 cycles.)
// Words of an operation: x0, x1, word of the sum, slot to clear | d0, d1, lane's slot, published slot | word to write.
template <int NB, int VS, bool BWD>
__device__ __forceinline__ void emo_spine_stage(unsigned op_a, unsigned n_bundles, unsigned slot_t, unsigned acc_t, unsigned G)
{
    uint4 s = emo_lds128(op_a), a = emo_lds128(op_a + 16u);
    unsigned to = emo_lds_u32(op_a + 32u);
    for (unsigned i = 0; i < n_bundles; ++i) {
        const EmoVec<VS> x0 = emo_ldv<VS>(slot_t + s.x * G), x1 = emo_ldv<VS>(slot_t + s.y * G), S = emo_ldv<VS>(acc_t + s.z * G);
        const uint4 c = a;
        const unsigned clear = s.w, dst = to;
        op_a += 48u * NB;
        s = emo_lds128(op_a);            // (behind the last bundle: a spare one)
        a = emo_lds128(op_a + 16u);
        to = emo_lds_u32(op_a + 32u);
        EmoVec<VS> q, y;
#pragma unroll
        for (int v = 0; v < VS; ++v) {
            q.v[v] = max(emo_floor_sub(x0.v[v], c.x), emo_floor_sub(x1.v[v], c.y));
            y.v[v] = q.v[v] + S.v[v];
        }
        emo_stv<VS>(slot_t + c.z * G, y);
        emo_stv<VS>(slot_t + c.w * G, y);
        emo_stv<VS>(acc_t + dst * G, BWD ? q : y);
        if (BWD) {
            EmoVec<VS> zero;
#pragma unroll
            for (int v = 0; v < VS; ++v) zero.v[v] = 0u;
            emo_stv<VS>(slot_t + clear * G, zero);
        }
        __syncwarp();                    // the next bundle's other threads read what this one stored
    }
}

// ---------------------------------------------------------------------------------------------------
// Forward pass (Eq. 1, Eq. 2): makespan and energy per policy, the restore list for the backward pass.
// ---------------------------------------------------------------------------------------------------
template <int VW, int VS, int NB, int MAXT>
__global__ void __launch_bounds__(MAXT, 1) emo_spine_fwd(SpineParams p)
{
    extern __shared__ __align__(128) unsigned char emo_smem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    constexpr int LP = 32 / NB;          // threads per operation
    const int G = p.groups, P = p.ptile, spines = P / (LP * VS), subs = G / VW;
    const int sub_op = lane / LP;        // spine: this thread's operation of a bundle
    const SpineRole role = emo_spine_role(p, warp, spines, false);
    const int64_t b0 = (int64_t)blockIdx.x * P;
    const int base_col = (p.want_base && p.B >= b0 && p.B < b0 + P) ? (int)(p.B - b0) : -1;
    const unsigned smem0 = emo_smem_addr(emo_smem), bar0 = smem0 + p.off_bar;
    volatile int *abort_word = reinterpret_cast<volatile int *>(emo_smem + p.off_bar + kBarKinds * kSpRing * 8);
    const long long limit = p.wait_cycles;
    emo_spine_init(p, emo_smem, bar0, spines, subs, false);
    emo_grid_wait_previous();            // (who wrote the levels; nothing in memory was touched so far)
    emo_grid_allow_next();               // the backward kernel's blocks may take SMs that are free: they read levels at once, and these are complete now

    long long T[VS];
    double ea[VW];
#pragma unroll
    for (int v = 0; v < VS; ++v) T[v] = 0;
#pragma unroll
    for (int v = 0; v < VW; ++v) ea[v] = 0.0;
    bool failed = false;
    if (role.prod) {
        emo_spine_produce<false>(p, smem0, bar0, abort_word, lane, role.idx);
    } else if (role.spine) {
        const unsigned word = (unsigned)((role.idx * LP + (lane & (LP - 1))) * VS);
        const unsigned slot_t = smem0 + word * 4u;
        long long t_pre = 0, t_loop = 0;
        SpineRing ra, rs;
        ra.n = p.nacc;
        rs.n = p.ns;
        const long long t_begin = EMO_SCLK();
        for (int c = 0; c < p.stages; ++c) {
            const long long tw0 = EMO_SCLK();
            if (!emo_spine_wait(emo_spine_bar(bar0, kBarSFull, rs.idx), rs.par, abort_word, limit) ||
                !emo_spine_wait(emo_spine_bar(bar0, kBarSums, ra.idx), ra.par, abort_word, limit)) {
                failed = true;
                break;
            }
            const long long tl0 = EMO_SCLK();
            t_pre += tl0 - tw0;
            const unsigned sta = smem0 + p.off_s0 + (unsigned)rs.idx * p.sbuf_bytes;
            const uint4 hd = emo_lds128(sta);          // bundles, terminal nodes
            emo_spine_stage<NB, VS, false>(sta + p.off_ops + 48u * (unsigned)sub_op, emo_uniform(hd.x), slot_t, smem0 + p.off_acc0 + (unsigned)ra.idx * p.acc_bytes + word * 4u, (unsigned)G);
            for (unsigned t = 0; t < hd.y; ++t) {
                // nodes without successors: candidates for the makespan
                const uint4 q = emo_lds128(sta + 16u + 16u * t);
                const EmoVec<VS> y = emo_ldv<VS>(slot_t + q.x * (unsigned)G);
                const long long lb = (long long)((unsigned long long)q.z | ((unsigned long long)q.w << 32));
#pragma unroll
                for (int v = 0; v < VS; ++v) T[v] = emo_max64(T[v], lb + (long long)(unsigned long long)y.v[v]);
            }
            t_loop += EMO_SCLK() - tl0;
            __syncwarp();
            if (lane == 0) {
                emo_mbar_arrive(emo_spine_bar(bar0, kBarSpine, ra.idx));
                emo_mbar_arrive(emo_spine_bar(bar0, kBarSEmpty, rs.idx));
            }
            ra.next();
            rs.next();
        }
        if (!failed && p.restore && sub_op == 0) {
            // the lanes' last values: where the completion walk begins
            uint32_t *const rst = p.restore + (size_t)blockIdx.x * p.restore_rows * P + word;
            for (int ln = 0; ln < p.lanes; ++ln)
                emo_stg_row_if<VS>(rst, (unsigned)p.pushes + (unsigned)ln, (unsigned)P * 4u, emo_ldv<VS>(slot_t + (unsigned)(ln * 128 * G)), 1u);
        }
        if (p.prof && lane == 0 && blockIdx.x < 512) {
            long long *pr = p.prof + ((size_t)blockIdx.x * 32 + warp) * 8;
            pr[0] = 0;
            pr[1] = t_pre;
            pr[2] = EMO_SCLK() - t_begin;
            pr[3] = t_loop;
        }
    } else if (role.post) {
        // The restore list: values that the spine left in the stage's words (a lane's value in front of a node whose start
        // does not follow from it alone), four at a time.
        const unsigned word = (unsigned)(role.idx * 32 * VW + lane * VW), P4 = (unsigned)P * 4u, G4 = (unsigned)G;
        uint32_t *const rst = p.restore + (size_t)blockIdx.x * p.restore_rows * P + word;
        SpineRing ra, rs;
        ra.n = p.nacc;
        rs.n = p.ns;
        for (int c = 0; c < p.stages; ++c) {
            if (!emo_spine_wait(emo_spine_bar(bar0, kBarSpine, ra.idx), ra.par, abort_word, limit) ||
                !emo_spine_wait(emo_spine_bar(bar0, kBarSFull, rs.idx), rs.par, abort_word, limit)) {
                failed = true;
                break;
            }
            const unsigned sta = smem0 + p.off_s0 + (unsigned)rs.idx * p.sbuf_bytes, acc_t = smem0 + p.off_acc0 + (unsigned)ra.idx * p.acc_bytes + word * 4u;
            const unsigned n = emo_uniform(emo_lds_u32(sta + 8u));          // records, a multiple of four
            for (unsigned i = 0; i < n; i += 4u) {
                const uint4 r0 = emo_lds128(sta + p.off_rec + 8u * i), r1 = emo_lds128(sta + p.off_rec + 8u * i + 16u);      // word, row; twice
                const unsigned w[4] = {r0.x, r0.z, r1.x, r1.z}, row[4] = {r0.y, r0.w, r1.y, r1.w};
                EmoVec<VW> y[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) y[k] = emo_ldv<VW>(acc_t + w[k] * G4);
#pragma unroll
                for (int k = 0; k < 4; ++k) emo_stg_row_if<VW>(rst, row[k], P4, y[k], row[k] + 1u);      // (kNone: padding)
            }
            __syncwarp();
            if (lane == 0) {
                emo_mbar_arrive(emo_spine_bar(bar0, kBarPost, ra.idx));
                emo_mbar_arrive(emo_spine_bar(bar0, kBarSEmpty, rs.idx));
            }
            ra.next();
            rs.next();
        }
    } else {
        failed = !emo_spine_look<VW, true>(p, smem0, bar0, abort_word, lane, role.idx, subs, base_col, p.posts ? kBarPost : kBarSpine, ea);
    }
    if (failed && lane == 0) {
        *abort_word = 1;
        if (p.status) atomicMin(p.status, -8);
    }

    // combine the workers of a sub-tile in a fixed order (run-to-run identical energy)
    __syncthreads();
    double *part = reinterpret_cast<double *>(emo_smem + p.off_w0);
    if (role.look)
#pragma unroll
        for (int v = 0; v < VW; ++v) part[(size_t)role.idx * 32 * VW + lane * VW + v] = ea[v];
    __syncthreads();
    if (role.spine && sub_op == 0 && !*abort_word) {
#pragma unroll
        for (int v = 0; v < VS; ++v) {
            const int col = emo_spine_policy<VW>((role.idx * LP + lane) * VS + v);
            const int64_t b = b0 + col;
            const int sub = col / (32 * VW), off = col - sub * 32 * VW;
            double e = 0.0;
            for (int k = 0; k < p.workers / subs; ++k) e += part[(size_t)(k * subs + sub) * 32 * VW + off];
            if (b < p.B) {
                p.makespan[b] = T[v];
                p.energy[b] = e;
            }
            if (base_col == col) {
                if (p.base_T) *p.base_T = T[v];
                if (p.base_E) *p.base_E = e;
            }
        }
    }
}

// ---------------------------------------------------------------------------------------------------
// Backward pass: slack of every node.  Stages are walked last to first.  The completion walk leaves the completion
// offset co of every segment, the spine its qin (the maximum over the successors of its last member); X = co + qin is
// one number for all members: slack = T - A - X.  The storing workers walk a segment's members last to first: the tail
// of a member is qin plus the durations up to it.  They write the slack and fold the tails behind the spine, which
// before a stage waits for the stores of the stage two back (folded values are read at least two stages
// after they are written).  EXTRA: also ES, LS, the slack sums and critical counts (ES_v = lbES_v + X - tail_v).
// ---------------------------------------------------------------------------------------------------
// Stores of this thread's V policies of one node.  VEC: they all exist and leave as one store.
template <int V, bool VEC>
__device__ __forceinline__ void emo_spine_put(const SpineParams &p, long long *base, unsigned row, unsigned ldo8, const long long (&x)[V], int64_t b, unsigned ok)
{
    if (VEC) {
        emo_stg_out_if<V>(base, row, ldo8, x, ok);
    } else {
#pragma unroll
        for (int v = 0; v < V; ++v) emo_stg_s64_if(base + v, row, ldo8, x[v], ok & (unsigned)(b + v < p.B));
    }
}
// The stores of one chunk, entries e0 .. e0 + n - 1 (n a multiple of four), everything taken for every member: without tails a
// member costs two loads per policy, the subtraction and its store.  EXTRA: with the tails, for ES, LS and the sums.
template <int V, bool VEC, bool EXTRA>
__device__ __forceinline__ void emo_spine_flat(const SpineParams &p, const EmoLevels<V> &lev, unsigned wbuf, unsigned acc_t, unsigned slot_t, unsigned e0, unsigned n,
                                               bool looks, const long long (&T)[V], int64_t b, long long (&ssum)[V], int (&ncrit)[V])
{
    constexpr int U = V == 4 ? (EXTRA ? 1 : 2) : (EXTRA ? 2 : 4);
    const unsigned P = (unsigned)p.ptile, P4 = P * 4u, G = (unsigned)p.groups, ldo8 = (unsigned)p.ldo * 8u, comp = p.comp_off * G;
    // entries without look-ups read the table row that stays zero
    const unsigned tab_row = looks ? p.tab_row : 0u, lvl_row = looks ? P : 0u;
    long long *const sl_t = p.slack ? reinterpret_cast<long long *>(p.slack) + b : nullptr;
    long long *const es_t = (EXTRA && p.ES) ? reinterpret_cast<long long *>(p.ES) + b : nullptr;
    long long *const ls_t = (EXTRA && p.LS) ? reinterpret_cast<long long *>(p.LS) + b : nullptr;
    const unsigned sl_ok = sl_t != nullptr, es_ok = es_t != nullptr, ls_ok = ls_t != nullptr;
    unsigned mem_a = wbuf + p.off_mem + e0 * 32u, lvl_a = wbuf + p.off_lvl + e0 * lvl_row, tab_a = wbuf + p.off_tab + (looks ? e0 : (unsigned)p.nlook) * p.tab_row;
    unsigned q[V], wn[U];
    uint4 mn[U], an[U];
    auto fetch = [&]() {
#pragma unroll
        for (int i = 0; i < U; ++i) {
            mn[i] = emo_lds128(mem_a + 32u * i);            // node, fold slot, fold correction, word << 16 | flags
            an[i] = emo_lds128(mem_a + 32u * i + 16u);      // A, lbES
            if (EXTRA) wn[i] = lev.load(lvl_a + (unsigned)i * lvl_row);
        }
        mem_a += 32u * U;
        lvl_a += lvl_row * U;
    };
    fetch();
#pragma unroll
    for (int v = 0; v < V; ++v) q[v] = 0;
    for (unsigned j0 = 0; j0 < n; j0 += U) {
        uint4 m[U], m2[U];
        unsigned d[U][V], qn[U][V], cn[U][V];
#pragma unroll
        for (int i = 0; i < U; ++i) {
            m[i] = mn[i];
            m2[i] = an[i];
            const unsigned at = acc_t + (m[i].w >> 16) * P4;
#pragma unroll
            for (int v = 0; v < V; ++v) {
                qn[i][v] = emo_lds_u32(at + 128u * v);
                cn[i][v] = emo_lds_u32(at + comp + 128u * v);
                if (EXTRA) d[i][v] = emo_lds_u32(lev.template addr<4u>(wn[i], v, tab_a + (unsigned)i * tab_row));
            }
        }
        fetch();                         // the next entries (past the last ones: read, not used)
        tab_a += tab_row * U;
#pragma unroll
        for (int i = 0; i < U; ++i) {
            const long long A = (long long)((unsigned long long)m2[i].x | ((unsigned long long)m2[i].y << 32));
            const unsigned real = (unsigned)(m[i].x != emo::kNone), slot = slot_t + m[i].y * G;
            long long sl[V];
            unsigned X[V];
#pragma unroll
            for (int v = 0; v < V; ++v) {
                X[v] = qn[i][v] + cn[i][v];
                sl[v] = (T[v] - A) - (long long)(unsigned long long)X[v];
            }
            emo_spine_put<V, VEC>(p, sl_t, m[i].x, ldo8, sl, b, sl_ok & real);
            if (EXTRA) {
                // ES_v = lbES_v + eo_v with eo_v = X - tail_v (X = eo + tail for every member)
                const long long lb = (long long)((unsigned long long)m2[i].z | ((unsigned long long)m2[i].w << 32));
                long long es[V], ls[V];
#pragma unroll
                for (int v = 0; v < V; ++v) {
                    q[v] = ((m[i].w & emo::kSpPos_First) ? qn[i][v] : q[v]) + d[i][v];
                    emo_red_max_u32(slot + 128u * v, emo_floor_sub(q[v], m[i].z));
                    es[v] = lb + (long long)(unsigned long long)(X[v] - q[v]);
                    ls[v] = es[v] + sl[v];
                    ssum[v] += real ? sl[v] : 0;
                    ncrit[v] += (real && sl[v] == 0) ? 1 : 0;
                }
                emo_spine_put<V, VEC>(p, es_t, m[i].x, ldo8, es, b, es_ok & real);
                emo_spine_put<V, VEC>(p, ls_t, m[i].x, ldo8, ls, b, ls_ok & real);
            }
        }
    }
}
// The same for slack alone where members are folded.  What is one number per segment is taken at its first member only: a bit per
// entry, made uniform once for up to 32 entries, says where (a branch on a freshly loaded word costs 100 cycles and more;
// taking everything for every member was 20 of the backward pass's 50 instructions per node and 32 policies).  Members that
// are not folded name a slot nobody reads.
template <int V, bool VEC>
__device__ __forceinline__ void emo_spine_folds(const SpineParams &p, const EmoLevels<V> &lev, unsigned wbuf, unsigned acc_t, unsigned slot_t, unsigned e0, unsigned n,
                                                bool looks, const long long (&T)[V], int64_t b)
{
    constexpr int U = V == 1 ? 4 : 2;
    const unsigned P = (unsigned)p.ptile, P4 = P * 4u, G = (unsigned)p.groups, ldo8 = (unsigned)p.ldo * 8u, comp = p.comp_off * G;
    const unsigned tab_row = looks ? p.tab_row : 0u, lvl_row = looks ? P : 0u;
    long long *const sl_t = p.slack ? reinterpret_cast<long long *>(p.slack) + b : nullptr;
    const unsigned sl_ok = sl_t != nullptr;
    unsigned mem_a = wbuf + p.off_mem + e0 * 32u, lvl_a = wbuf + p.off_lvl + e0 * lvl_row, tab_a = wbuf + p.off_tab + (looks ? e0 : (unsigned)p.nlook) * p.tab_row;
    unsigned q[V], wn[U], first = 0;
    long long sl[V];
    uint4 mn[U];
    auto fetch = [&]() {
#pragma unroll
        for (int i = 0; i < U; ++i) {
            mn[i] = emo_lds128(mem_a + 32u * i);            // node, fold slot, fold correction, word << 16 | flags
            wn[i] = lev.load(lvl_a + (unsigned)i * lvl_row);
        }
        lvl_a += lvl_row * U;
    };
    fetch();
#pragma unroll
    for (int v = 0; v < V; ++v) {
        q[v] = 0;
        sl[v] = 0;
    }
    for (unsigned e = e0; e < e0 + n; e += U) {
        if (e == e0 || (e & 31u) == 0u) first = emo_uniform(emo_lds_u32(wbuf + p.off_first + (e >> 5) * 4u)) >> (e & 31u);
        const unsigned rec_a = mem_a;
        uint4 m[U];
        unsigned d[U][V];
#pragma unroll
        for (int i = 0; i < U; ++i) {
            m[i] = mn[i];
#pragma unroll
            for (int v = 0; v < V; ++v) d[i][v] = emo_lds_u32(lev.template addr<4u>(wn[i], v, tab_a + (unsigned)i * tab_row));
        }
        mem_a += 32u * U;
        tab_a += tab_row * U;
        fetch();                         // the next entries (past the last ones: read, not used)
#pragma unroll
        for (int i = 0; i < U; ++i) {
            if (first & (1u << i)) {
                const EmoVec<2> a = emo_ldv<2>(rec_a + 32u * i + 16u);
                const unsigned at = acc_t + (m[i].w >> 16) * P4;
                const long long A = (long long)((unsigned long long)a.v[0] | ((unsigned long long)a.v[1] << 32));
#pragma unroll
                for (int v = 0; v < V; ++v) {
                    q[v] = emo_lds_u32(at + 128u * v);
                    sl[v] = (T[v] - A) - (long long)(unsigned long long)(q[v] + emo_lds_u32(at + comp + 128u * v));
                }
            }
            const unsigned slot = slot_t + m[i].y * G;
            emo_spine_put<V, VEC>(p, sl_t, m[i].x, ldo8, sl, b, sl_ok & (unsigned)(m[i].x != emo::kNone));
#pragma unroll
            for (int v = 0; v < V; ++v) {
                q[v] += d[i][v];
                emo_red_max_u32(slot + 128u * v, emo_floor_sub(q[v], m[i].z));
            }
        }
        first >>= U;
    }
}

template <int VW, int VS, int NB, int MAXT, bool EXTRA>
__global__ void __launch_bounds__(MAXT, 1) emo_spine_bwd(SpineParams p)
{
    extern __shared__ __align__(128) unsigned char emo_smem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    constexpr int LP = 32 / NB;          // threads per operation
    const int G = p.groups, P = p.ptile, spines = P / (LP * VS), subs = G / VW;
    const int sub_op = lane / LP;        // spine: this thread's operation of a bundle
    const SpineRole role = emo_spine_role(p, warp, spines, true);
    const int64_t b0 = (int64_t)blockIdx.x * P;
    const unsigned smem0 = emo_smem_addr(emo_smem), bar0 = smem0 + p.off_bar;
    volatile int *abort_word = reinterpret_cast<volatile int *>(emo_smem + p.off_bar + kBarKinds * kSpRing * 8);
    const long long limit = p.wait_cycles;
    emo_grid_allow_next();
    emo_spine_init(p, emo_smem, bar0, spines, subs, true);
    // everything but the first loads of level rows and tables waits for the forward kernel (which has waited for the levels when
    // this one starts)
    if (!(role.prod && role.idx == 0)) emo_grid_wait_previous();

    bool failed = false;
    long long ssum[VW];
    int ncrit[VW];
#pragma unroll
    for (int v = 0; v < VW; ++v) {
        ssum[v] = 0;
        ncrit[v] = 0;
    }
    if (role.prod) {
        emo_spine_produce<true>(p, smem0, bar0, abort_word, lane, role.idx);
    } else if (role.spine) {
        const unsigned word4 = (unsigned)((role.idx * LP + (lane & (LP - 1))) * VS) * 4u;
        long long t_pre = 0, t_loop = 0;
        SpineRing ra, rs, ra2;
        ra.n = ra2.n = p.nacc;
        rs.n = p.ns;
        const long long t_begin = EMO_SCLK();
        for (int c = 0; c < p.stages; ++c) {
            const long long tw0 = EMO_SCLK();
            // staged operations; completion offsets (and with them the sums); from the third stage on the stores of stage c - 2
            const bool third = c >= 2;
            if (!emo_spine_wait(emo_spine_bar(bar0, kBarSFull, rs.idx), rs.par, abort_word, limit) ||
                !emo_spine_wait(emo_spine_bar(bar0, kBarComp, ra.idx), ra.par, abort_word, limit) ||
                (third && !emo_spine_wait(emo_spine_bar(bar0, kBarPost, ra2.idx), ra2.par, abort_word, limit))) {
                failed = true;
                break;
            }
            if (third) ra2.next();
            const long long tw3 = EMO_SCLK();
            t_pre += tw3 - tw0;
            const unsigned sta = smem0 + p.off_s0 + (unsigned)rs.idx * p.sbuf_bytes;
            emo_spine_stage<NB, VS, true>(sta + p.off_ops + 48u * (unsigned)sub_op, emo_uniform(emo_lds_u32(sta)), smem0 + word4, smem0 + p.off_acc0 + (unsigned)ra.idx * p.acc_bytes + word4, (unsigned)G);
            t_loop += EMO_SCLK() - tw3;
            __syncwarp();
            if (lane == 0) {
                emo_mbar_arrive(emo_spine_bar(bar0, kBarSpine, ra.idx));
                emo_mbar_arrive(emo_spine_bar(bar0, kBarSEmpty, rs.idx));
            }
            ra.next();
            rs.next();
        }
        if (p.prof && lane == 0 && blockIdx.x < 512) {
            long long *pr = p.prof + ((size_t)blockIdx.x * 32 + warp) * 8;
            pr[0] = 0;
            pr[1] = t_pre;
            pr[2] = EMO_SCLK() - t_begin;
            pr[3] = t_loop;
        }
    } else if (role.comp) {
        // The completion offsets: per lane and stage the segments last to first.  co of a segment's last member is what the
        // segment behind it started from: that segment's co minus its sum, or a word of the restore list.  The lanes are dealt
        // to NB streams, one for every part of the warp; R records at a time (what the registers hold without spilling: with
        // the shared memory in use there is hardly any L1, a spilled word comes back from L2).
        constexpr int R = VS == 4 ? 2 : 4;
        const unsigned word = (unsigned)((role.idx * LP + (lane & (LP - 1))) * VS), P4 = (unsigned)P * 4u, G4 = (unsigned)G, comp = p.comp_off * G4;
        const unsigned slot_t = smem0 + word * 4u;
        for (int ln = 0; ln < p.lanes; ++ln) {
            const uint32_t *src = p.restore + ((size_t)blockIdx.x * p.restore_rows + p.pushes + ln) * P + word;
            EmoVec<VS> y;
#pragma unroll
            for (int v = 0; v < VS; ++v) y.v[v] = src[v];
            if (sub_op == 0) emo_stv<VS>(slot_t + (unsigned)(p.c_slot0 + ln) * 128u * G4, y);
        }
        __syncwarp();
        long long t_pre = 0, t_loop = 0;
        SpineRing ra, rs;
        ra.n = p.nacc;
        rs.n = p.ns;
        const long long t_begin = EMO_SCLK();
        for (int c = 0; c < p.stages; ++c) {
            const long long tw0 = EMO_SCLK();
            if (!emo_spine_wait(emo_spine_bar(bar0, kBarSFull, rs.idx), rs.par, abort_word, limit) ||
                !emo_spine_wait(emo_spine_bar(bar0, kBarSums, ra.idx), ra.par, abort_word, limit)) {
                failed = true;
                break;
            }
            const long long tw1 = EMO_SCLK();
            t_pre += tw1 - tw0;
            const unsigned sta = smem0 + p.off_s0 + (unsigned)rs.idx * p.sbuf_bytes;
            const unsigned acc_t = smem0 + p.off_acc0 + (unsigned)ra.idx * p.acc_bytes + word * 4u, rst_a = sta + p.off_rst + word * 4u;
            unsigned rec_a = sta + p.off_rec + 16u * (unsigned)sub_op;
            const unsigned n = emo_uniform(emo_lds_u32(sta + 8u));          // records of a stream, a multiple of four
            EmoVec<VS> co;
#pragma unroll
            for (int v = 0; v < VS; ++v) co.v[v] = 0u;
            for (unsigned i = 0; i < n; i += R) {
                uint4 r[R];
                EmoVec<VS> S[R], in[R], pop[R];
#pragma unroll
                for (int k = 0; k < R; ++k) r[k] = emo_lds128(rec_a + 16u * NB * k);      // the lane's slot, word of the sum, word of the segment, flags
                rec_a += 16u * NB * R;
#pragma unroll
                for (int k = 0; k < R; ++k) {
#pragma unroll
                    for (int v = 0; v < VS; ++v) pop[k].v[v] = 0u;
                    S[k] = emo_ldv<VS>(acc_t + r[k].y * G4);
                    in[k] = emo_ldv<VS>(slot_t + r[k].x * G4);
                    emo_ldv_if<VS>(pop[k], rst_a + (r[k].w >> 8) * P4, r[k].w & emo::kSpDev_Pop);
                }
#pragma unroll
                for (int k = 0; k < R; ++k) {
#pragma unroll
                    for (int v = 0; v < VS; ++v) co.v[v] = (r[k].w & emo::kSpPos_First) ? in[k].v[v] : co.v[v];
                    emo_stv<VS>(acc_t + r[k].z * G4 + comp, co);
#pragma unroll
                    for (int v = 0; v < VS; ++v) co.v[v] = (r[k].w & emo::kSpDev_Pop) ? pop[k].v[v] : co.v[v] - S[k].v[v];
                    emo_stv_if<VS>(slot_t + r[k].x * G4, co, r[k].w & emo::kSpPos_Last);
                }
            }
            t_loop += EMO_SCLK() - tw1;
            __syncwarp();
            if (lane == 0) {
                emo_mbar_arrive(emo_spine_bar(bar0, kBarComp, ra.idx));
                emo_mbar_arrive(emo_spine_bar(bar0, kBarSEmpty, rs.idx));
            }
            ra.next();
            rs.next();
        }
        if (p.prof && lane == 0 && blockIdx.x < 512) {
            long long *pr = p.prof + ((size_t)blockIdx.x * 32 + warp) * 8;
            pr[0] = 0;
            pr[1] = t_pre;
            pr[2] = EMO_SCLK() - t_begin;
            pr[3] = t_loop;
        }
    } else if (role.look) {
        double none[VW];
        failed = !emo_spine_look<VW, false>(p, smem0, bar0, abort_word, lane, role.idx, subs, -1, kBarPost, none);
    } else {
        const int sub = role.idx % subs, np = p.posts / subs;
        EmoLevels<VW> lev;
        lev.init(p, sub, lane, -1);
        const int64_t b = b0 + sub * 32 * VW + lane * VW;
        const bool vec = VW > 1 && p.vec_out && b0 + (sub + 1) * 32 * VW <= p.B;
        long long T[VW];
#pragma unroll
        for (int v = 0; v < VW; ++v) T[v] = b + v < p.B ? p.makespan[b + v] : 0;
        const unsigned col = (unsigned)(sub * 32 * VW + lane) * 4u;
        long long t_w = 0, t_work = 0;
        SpineRing rw, ra;
        rw.n = p.nw;
        ra.n = p.nacc;
        const long long t_begin = EMO_SCLK();
        for (int c = 0, chunk = role.idx / subs;; chunk += np) {
            for (; chunk >= p.chunks_post; chunk -= p.chunks_post, ++c) {
                rw.next();
                ra.next();
            }
            if (c >= p.stages) break;
            const long long tw0 = EMO_SCLK();
            // (the spine's results imply the staged data; their barrier is read too because the copies signal there)
            if (!emo_spine_wait(emo_spine_bar(bar0, kBarSpine, ra.idx), ra.par, abort_word, limit) ||
                !emo_spine_wait(emo_spine_bar(bar0, kBarWFull, rw.idx), rw.par, abort_word, limit)) {
                failed = true;
                break;
            }
            const long long tw1 = EMO_SCLK();
            t_w += tw1 - tw0;
            const unsigned wbuf = smem0 + p.off_w0 + (unsigned)rw.idx * p.wbuf_bytes, acc_t = smem0 + p.off_acc0 + (unsigned)ra.idx * p.acc_bytes + col;
            const unsigned ck = emo_uniform(emo_lds_u32(wbuf + 4u * (unsigned)(kSpChunks + chunk))), e0 = ck & 0xFFFFu, n = (ck >> 16) & 0x7FFFu;
            const bool looks = chunk < p.chunks;
            if (!EXTRA && (ck >> 31)) {
                if (vec) emo_spine_folds<VW, true>(p, lev, wbuf, acc_t, smem0 + col, e0, n, looks, T, b);
                else emo_spine_folds<VW, false>(p, lev, wbuf, acc_t, smem0 + col, e0, n, looks, T, b);
            } else {
                if (vec) emo_spine_flat<VW, true, EXTRA>(p, lev, wbuf, acc_t, smem0 + col, e0, n, looks, T, b, ssum, ncrit);
                else emo_spine_flat<VW, false, EXTRA>(p, lev, wbuf, acc_t, smem0 + col, e0, n, looks, T, b, ssum, ncrit);
            }
            __syncwarp();
            if (lane == 0) {
                emo_mbar_arrive(emo_spine_bar(bar0, kBarPost, ra.idx));
                emo_mbar_arrive(emo_spine_bar(bar0, kBarWEmpty, rw.idx));
            }
            t_work += EMO_SCLK() - tw1;
        }
        if (p.prof && lane == 0 && blockIdx.x < 512) {
            long long *pr = p.prof + ((size_t)blockIdx.x * 32 + warp) * 8;
            pr[0] = 0;
            pr[1] = t_w;
            pr[2] = EMO_SCLK() - t_begin;
            pr[4] = t_work;
        }
    }
    if (failed && lane == 0) {
        *abort_word = 1;
        if (p.status) atomicMin(p.status, -8);
    }
    if (EXTRA) {
        // per-policy sums: the storing workers' parts combined in their order
        __syncthreads();
        long long *part = reinterpret_cast<long long *>(emo_smem + p.off_w0);
        if (role.post) {
#pragma unroll
            for (int v = 0; v < VW; ++v) {
                long long *pd = part + ((size_t)role.idx * 32 * VW + lane * VW + v) * 2;
                pd[0] = ssum[v];
                pd[1] = (long long)ncrit[v];
            }
        }
        __syncthreads();
        if (!*abort_word)
            for (int col = threadIdx.x; col < P; col += blockDim.x) {
                const int64_t b = b0 + col;
                const int sub = col / (32 * VW), off = col - sub * 32 * VW;
                long long s2 = 0, cnt = 0;
                for (int k = 0; k < p.posts / subs; ++k) {
                    s2 += part[((size_t)(k * subs + sub) * 32 * VW + off) * 2];
                    cnt += part[((size_t)(k * subs + sub) * 32 * VW + off) * 2 + 1];
                }
                if (b < p.B) {
                    if (p.slack_sum) p.slack_sum[b] = s2;
                    if (p.n_critical) p.n_critical[b] = (int32_t)cnt;
                }
            }
    }
}
#undef EMO_SCLK
