// C-ABI entry points (see include/emo.h) and the CUDA kernels behind them.  sm_100a only.
#include <cuda_runtime.h>

#include <algorithm>
#include <chrono>
#include <cmath>
#include <cstdio>
#include <map>
#include <cstring>
#include <new>
#include <string>
#include <thread>
#include <vector>

#include "../../include/emo.h"
#include "emo_compile.h"
#include "emo_contract.h"
#include "emo_flow.h"
#include "emo_kernels.cuh"
#include "emo_pass_lane.cuh"
#include "emo_pass_staged.cuh"
#include "emo_flow.cuh"
#include "emo_spine.cuh"
#include "emo_intervals.cuh"
#include "emo_model.cuh"
#include "emo_generic.cuh"
#include "emo_slice.cuh"
#include "emo_walk.cuh"

using namespace emo;

struct DevProgram {
    unsigned char *rec = nullptr;   // records: entry, duration row, (forward) energy row
    uint32_t *rows = nullptr;
    uint32_t *groups = nullptr;     // the nodes' groups (time-interval policies)
    int rec_bytes = 0;
};

// The same program in the layout of emo_pass_lane (see emo_lane_layout.cuh), padded to whole stages.
struct DevProgramLane {
    unsigned char *ent = nullptr;   // [Qp][32]
    unsigned char *tab = nullptr;   // [Qp][tab_entry]
    uint32_t *rows = nullptr;       // [Qp]
    int steps_pad = 0;
    unsigned tab_entry = 0;
};

// The lane-stream program on the device: one blob per stage and direction (see emo_flow.cuh).
struct DevFlow {
    unsigned char *blobF = nullptr, *blobB = nullptr;
    unsigned char *blobFI = nullptr;      // the forward blob followed by 32 bytes per entry: time-interval policies
    uint32_t *rows = nullptr, *push_base = nullptr;
    unsigned blobF_bytes = 0, blobB_bytes = 0, blobFI_bytes = 0, f_off_meta = 0;
    int64_t packs = 0, switches = 0;      // time-interval policies: entries with a policy, and those whose predecessor on the lane is another device's
    unsigned off_seg = 0;
    unsigned f_off_rec = 0, f_off_pool = 0, f_off_tab = 0;
    unsigned b_off_rec = 0, b_off_pool = 0, b_off_lbes = 0, b_off_tab = 0;
    int max_push = 0;               // most restore rows of one stage
    bool ready = false;
};

// The spine program on the device (emo_spine.cuh): per direction and stage the workers' part and the spine's part.
struct DevSpineDir {
    unsigned char *blobW = nullptr, *blobS = nullptr;
    uint32_t *rows = nullptr;       // [stages][nlook] policy row of every look-up entry
    unsigned w_bytes = 0, s_bytes = 0, off_pos = 0, off_mem = 0, off_first = 0, off_tab = 0, off_ops = 0, off_rec = 0;
    int words = 0;                  // words per policy and stage: sums (later the values that are pushed / qin), one that stays zero, an unread one; backward then
                                    // the completion offsets
    int zero = 0;                   // the word that stays zero
};
struct DevSpine {
    DevSpineDir f, b;
    unsigned char *mem = nullptr;   // the allocation that holds all of it
    uint32_t *push_base = nullptr;
    int nlook = 0, chunks = 0;      // look-up entries and chunks of a stage
    int max_push = 0;
    bool ready = false;             // on the device (host-only handles: laid out)
};

// Blocks of the slice kernels: policies, slices.
constexpr int kSliceShapes = 3;
constexpr int kSliceP[kSliceShapes] = {1, 8, 16}, kSliceS[kSliceShapes] = {4, 1, 1};

// The slice program on the device (emo_slice.cuh), and what its launches need to know.
struct DevSlice {
    unsigned char *mem = nullptr;   // the allocation that holds all of it
    uint32_t *blob = nullptr;
    uint4 *index = nullptr, *rec = nullptr;
    uint32_t *tabT = nullptr;
    double *tabE = nullptr;
    int count = 0, cols = 0, Lp = 0, group = 0, groups = 0;
    unsigned head = 0, words = 0, steps[2] = {0, 0}, nodes = 0, len[2] = {0, 0};      // most of one slice
    unsigned slots1[2] = {0, 0}, slots2[2] = {0, 0};
    bool ready = false;
};

// The spine program as the device gets it: one allocation, one copy.
struct SpineImage {
    std::vector<unsigned char> host;
    size_t at_fW = 0, at_fS = 0, at_bW = 0, at_bS = 0, at_rowsF = 0, at_rowsB = 0, at_pb = 0;
};

struct emo_graph {
    HostGraph h;
    Program fwd, bwd;
    Flow flow;                       // lane-stream program of the 32-bit pass kernels (flow.ok32: usable)
    DevProgram dfwd, dbwd;
    DevProgramLane lfwd, lbwd;       // only for programs of at most kLaneMaxLanes lanes
    DevFlow dflow;
    Flow sflow;                      // the same graph compiled with short stages and its spine program (sflow.spine.ok: usable)
    DevSpine dspine;
    Flow lflow;                      // ... and once more with longer stages, for calls of at most two policy groups per SM
    DevSpine dlong;
    DevSlice dslice;                 // slices of the graph, for calls with few policies
    SpineImage simage, limage;       // both as laid out for the device (kept by host-only handles, else until they are copied)
    Walk walk;                       // time-interval policies (EMO_F_INTERVALS), a thread per policy; its blob is kept on the device
    unsigned char *dwalk = nullptr;
    emo_graph *joined = nullptr;     // the contracted graph (emo_contract.h) that emo_eval_policies evaluates; null where it saves little
    bool host_only = false;
    // graphs beyond the schedule compilers' limits (or loaded with EMO_F_GENERIC): evaluated by the generic kernels
    bool generic = false;
    int64_t *gen_row_ptr = nullptr, *gen_srow_ptr = nullptr, *gen_lat = nullptr;
    int32_t *gen_col = nullptr, *gen_scol = nullptr, *gen_group = nullptr;
    double *gen_energy = nullptr;
    std::vector<int64_t> host_lat;      // kept only for the generic path's upload
    std::vector<double> host_energy;
    size_t one_bytes = 0;            // workspace that emo_slack asks for
    int device = 0;
    int sm_count = 148;
    size_t smem_optin = 0;
};

namespace {

constexpr int kManySlots = 48;       // above this, a program is compiled with the short barrier distance
constexpr size_t kSmallWs = 65536;   // head of the workspace: selection partials and scalars

// Optional timing hook: events recorded around the forward and the backward pass kernel.
cudaEvent_t g_pass_events[4] = {nullptr, nullptr, nullptr, nullptr};

size_t round_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

// workspace area for one policy's levels laid out [rows][16] (row pitch a bulk copy accepts)
size_t lvl_area(const emo_graph *g);

#define EMO_CUDA(call)                                  \
    do {                                                \
        cudaError_t e_ = (call);                        \
        if (e_ != cudaSuccess) { (void)cudaGetLastError(); return EMO_E_CUDA; } \
    } while (0)

template <typename T>
int upload(T **dst, const void *src, size_t bytes)
{
    *dst = nullptr;
    if (bytes == 0) bytes = 16;
    if (cudaMalloc((void **)dst, bytes) != cudaSuccess) { (void)cudaGetLastError(); *dst = nullptr; return EMO_E_OOM; }
    if (src && cudaMemcpy(*dst, src, bytes, cudaMemcpyHostToDevice) != cudaSuccess) { (void)cudaGetLastError(); return EMO_E_CUDA; }
    return EMO_OK;
}

int upload_program(const Program &p, DevProgram &d)
{
    const size_t Q = (size_t)p.steps * p.lanes;
    const bool fwd = !p.energy.empty();
    d.rec_bytes = 32 + p.Lp * 4 + (fwd ? p.Lp * 8 : 0);
    std::vector<unsigned char> rec(Q * d.rec_bytes);
    for (size_t q = 0; q < Q; ++q) {
        unsigned char *r = rec.data() + q * d.rec_bytes;
        std::memcpy(r, &p.entries[q * kEntryWords], 32);
        std::memcpy(r + 32, &p.lat[q * p.Lp], (size_t)p.Lp * 4);
        if (fwd) std::memcpy(r + 32 + p.Lp * 4, &p.energy[q * p.Lp], (size_t)p.Lp * 8);
    }
    int rc = upload(&d.rec, rec.data(), rec.size());
    if (rc) return rc;
    rc = upload(&d.rows, p.rows.data(), p.rows.size() * sizeof(uint32_t));
    if (rc) return rc;
    return upload(&d.groups, p.groups.data(), p.groups.size() * sizeof(uint32_t));
}

int upload_program_lane(const Program &p, DevProgramLane &d)
{
    const bool fwd = !p.energy.empty();
    const size_t Q = (size_t)p.steps * p.lanes;
    d.steps_pad = (p.steps + kLaneStepPad - 1) / kLaneStepPad * kLaneStepPad;
    const size_t Qp = (size_t)d.steps_pad * p.lanes;
    d.tab_entry = (unsigned)p.Lp * (fwd ? 12u : 4u);
    std::vector<uint32_t> ent(Qp * 8, 0), rows(Qp, kNone);
    std::vector<unsigned char> tab(Qp * d.tab_entry, 0);
    for (size_t q = 0; q < Qp; ++q) {
        uint32_t *w = &ent[q * 8];
        w[0] = kNone;
        w[1] = kLaneNoSlot | kLaneIdle;
        w[2] = 0xFFFFFFFFu;      // idle: the lane keeps its value
        w[5] = kNone;
        if (q >= Q) continue;
        const uint32_t *en = &p.entries[q * kEntryWords];
        const uint32_t fl = en[1];
        if (!(fl & kValid)) {
            w[1] |= (en[5] & 15u) << kLaneRunShift;      // forward: an idle entry may sit inside a run
            continue;
        }
        const uint32_t np = (fl >> kNPredShift) & 7u;
        const uint32_t out = (fl & kWriteSlot) ? ((fl >> kOutShift) & 255u) : kLaneNoSlot;
        const uint32_t outpar = (fl & kWriteSlot) ? ((fl >> kOutParityShift) & 1u) : 0u;
        const uint32_t oppar = (fl >> kOperandParityShift) & 63u;
        w[0] = en[0];
        w[1] = out | (np << kLaneNpShift) | ((fl & kTerminal) ? kLaneTerminal : 0u) | (outpar << kLaneOutParShift) | (oppar << kLaneOpParShift);
        w[1] |= (en[5] & 15u) << kLaneRunShift;
        if (en[6] & 1u) w[1] |= kLaneSettled;
        w[2] = (fl & kRegPred) ? 0xFFFFFFFFu : 0u;
        w[3] = en[2];
        w[4] = en[3];
        w[5] = en[4];
        rows[q] = p.rows[q];
        // a node that ignores the policy (level mask 0) gets its level-0 value at every index:
        // the kernel indexes the row with whatever byte it finds
        const bool uses_level = ((fl >> kMaskShift) & 255u) != 0;
        for (int l = 0; l < p.Lp; ++l) {
            const size_t src = q * p.Lp + (uses_level ? l : 0);
            unsigned char *t = tab.data() + q * d.tab_entry + (size_t)l * (fwd ? 12 : 4);
            std::memcpy(t, &p.lat[src], 4);
            if (fwd) {
                uint64_t bits;
                std::memcpy(&bits, &p.energy[src], 8);
                const uint32_t hi = (uint32_t)(bits >> 32), lo = (uint32_t)bits;
                std::memcpy(t + 4, &hi, 4);
                std::memcpy(t + 8, &lo, 4);
            }
        }
    }
    int rc = upload(&d.ent, ent.data(), ent.size() * 4);
    if (rc == EMO_OK) rc = upload(&d.tab, tab.data(), tab.size());
    if (rc == EMO_OK) rc = upload(&d.rows, rows.data(), rows.size() * 4);
    return rc;
}

void free_program_lane(DevProgramLane &d)
{
    if (d.ent) cudaFree(d.ent);
    if (d.tab) cudaFree(d.tab);
    if (d.rows) cudaFree(d.rows);
    d = DevProgramLane();
}

void free_program(DevProgram &d)
{
    if (d.rec) cudaFree(d.rec);
    if (d.rows) cudaFree(d.rows);
    if (d.groups) cudaFree(d.groups);
    d = DevProgram();
}

// Longest path with one duration per node (used for the overflow guard and the info block).
template <typename F>
__int128 host_longest(const HostGraph &h, F dur)
{
    std::vector<__int128> C((size_t)std::max(h.n, 1));
    __int128 T = 0;
    for (int32_t v = 0; v < h.n; ++v) {
        __int128 s = 0;
        for (int64_t e = h.row_ptr[v]; e < h.row_ptr[v + 1]; ++e) s = std::max(s, C[h.col[e]]);
        C[v] = s + dur(v);
        T = std::max(T, C[v]);
    }
    return T;
}

size_t lvl_area(const emo_graph *g) { return round_up((size_t)std::max(g->h.rows, 1) * 16, 256); }

struct LaunchShape {
    int groups, grid, threads;
    size_t smem;
};

// Policy groups (32 policies each) per block: enough to give every SM one block, bounded by the
// block size, the named barriers (ids 1..15) and shared memory.
int shape_for(const emo_graph *g, const Program &p, int64_t NB, LaunchShape &s)
{
    int64_t n_groups = (NB + 31) / 32;
    int gmax = std::min(32 / p.lanes, 15);
    if (gmax < 1) return EMO_E_UNSUPPORTED;
    size_t per_group = (size_t)p.slots * 256 + (size_t)p.lanes * 32 * 16;
    size_t budget = g->smem_optin ? g->smem_optin : 48 * 1024;
    while (gmax > 1 && per_group * gmax > budget) --gmax;
    if (per_group * gmax > budget) return EMO_E_UNSUPPORTED;
    int64_t want = (n_groups + g->sm_count - 1) / g->sm_count;
    s.groups = (int)std::max<int64_t>(1, std::min<int64_t>(gmax, want));
    s.grid = (int)((n_groups + s.groups - 1) / s.groups);
    s.threads = s.groups * p.lanes * 32;
    s.smem = per_group * s.groups;
    return EMO_OK;
}

// Shape of the staged kernel: groups of 64 policies (two per thread), one more warp produces, then
// as many steps per stage as fit beside the slots.  Returns false when it cannot be used.
bool staged_shape(const emo_graph *g, const Program &p, int rec_bytes, bool backward, int64_t NB, LaunchShape &s,
                  StagedParams &sp)
{
    if (p.steps == 0 || !g->smem_optin) return false;
    int64_t n_groups = (NB + 63) / 64;
    int gmax = std::min((32 - kProducerWarps) / p.lanes, 15);
    if (gmax < 1) return false;
    int64_t want = (n_groups + g->sm_count - 1) / g->sm_count;
    int G = (int)std::max<int64_t>(1, std::min<int64_t>(gmax, want));
    const size_t budget = g->smem_optin;
    static const int kTry[5][2] = {{16, 4}, {16, 3}, {8, 4}, {8, 3}, {8, 2}};   // {steps per stage, stages}
    for (; G >= 1; --G) {
        const size_t P = 64 * (size_t)G;
        const size_t fixed = (size_t)G * p.slots * kSlotStride + (size_t)G * p.lanes * 1024 + 256 + 128;
        for (int t = 0; t < 5; ++t) {
            const int sc = kTry[t][0], stages = kTry[t][1];
            const size_t ne = (size_t)sc * p.lanes;
            if (ne > 32 * (size_t)kRowRegs) continue;
            const size_t stage_bytes = round_up(ne * ((size_t)rec_bytes + P + (backward ? P * 8 : 0)), 128);
            if (fixed + stages * stage_bytes > budget) continue;
            sp.sc = sc;
            sp.stages = stages;
            sp.ptile = (int)P;
            sp.off_lvl = (unsigned)(ne * rec_bytes);
            sp.off_es = sp.off_lvl + (unsigned)(ne * P);
            sp.stage_bytes = (unsigned)stage_bytes;
            sp.off_part = (unsigned)round_up((size_t)G * p.slots * kSlotStride, 16);
            sp.off_bar = sp.off_part + (unsigned)((size_t)G * p.lanes * 1024);
            sp.off_stage0 = (unsigned)round_up(sp.off_bar + 256, 128);
            s.groups = G;
            s.grid = (int)((n_groups + G - 1) / G);
            s.threads = (G * p.lanes + kProducerWarps) * 32;
            s.smem = sp.off_stage0 + (size_t)stages * sp.stage_bytes;
            if (s.smem > budget) continue;
            return true;
        }
    }
    return false;
}

// Shape of the kernel with one warp per schedule lane and one policy per thread: groups of 32
// policies, one more warp produces; slot area, partial results, barriers, then the stage ring.
bool lane_shape(const emo_graph *g, const Program &p, bool backward, int64_t NB, LaunchShape &s, StagedParams &sp)
{
    if (p.steps == 0 || !g->smem_optin || !g->lfwd.ent || !g->lbwd.ent) return false;
    const size_t rec_bytes = 32 + (size_t)p.Lp * (backward ? 4 : 12);     // entry and table row
    const int64_t n_groups = (NB + 31) / 32;
    const int gmax = std::min((32 - kProducerWarps) / p.lanes, 15);
    if (gmax < 1) return false;
    const int64_t want = (n_groups + g->sm_count - 1) / g->sm_count;
    int G = (int)std::max<int64_t>(1, std::min<int64_t>(gmax, want));
    const size_t budget = g->smem_optin;
    // {steps per stage, stages}: long stages first - a stage boundary costs every warp about a
    // microsecond (measured: 8, 16, 32 steps per stage gave 15.1, 12.3, 11.4 ms on the same forward
    // pass), while two stages hide the refill as well as four
    static const int kTry[10][2] = {{32, 2}, {16, 3}, {16, 2}, {8, 3}, {8, 2}, {4, 6}, {4, 5}, {4, 4}, {4, 3}, {4, 2}};
    for (; G >= 1; --G) {
        const size_t P = 32 * (size_t)G;
        const size_t slot_bytes = round_up((size_t)G * p.slots * kLaneSlotStride, 16);
        const size_t part_bytes = (size_t)G * p.lanes * 32 * 16;
        const size_t head = round_up(slot_bytes + part_bytes + 256, 128);
        for (int t = 0; t < 10; ++t) {
            const int sc = kTry[t][0], stages = kTry[t][1];
            const size_t ne = (size_t)sc * p.lanes;
            if (ne > 32 * (size_t)kRowRegs || stages > kMaxStages || kLaneStepPad % sc != 0) continue;
            const size_t stage_bytes = round_up(ne * (rec_bytes + P + (backward ? P * 8 : 0)), 128);
            // behind the last stage: room for the look-ahead of its last step
            const size_t pad = round_up((size_t)p.lanes * std::max<size_t>(P * 8, rec_bytes), 128);
            const size_t total = head + stages * stage_bytes + pad;
            if (total > budget) continue;
            sp.sc = sc;
            sp.stages = stages;
            sp.ptile = (int)P;
            sp.off_lvl = (unsigned)(ne * rec_bytes);
            sp.off_es = sp.off_lvl + (unsigned)(ne * P);
            sp.stage_bytes = (unsigned)stage_bytes;
            sp.off_part = (unsigned)slot_bytes;
            sp.off_bar = (unsigned)(slot_bytes + part_bytes);
            sp.off_stage0 = (unsigned)head;
            s.groups = G;
            s.grid = (int)((n_groups + G - 1) / G);
            s.threads = (G * p.lanes + kProducerWarps) * 32;
            s.smem = total;
            return true;
        }
    }
    return false;
}

// How the two passes of one call will run: both staged (earliest starts travel through the tiled
// spill) or both with the plain kernels (through an [n][ldes] array).
struct PassPlan {
    bool staged = false;
    bool lane_f = false, lane_b = false;   // staged, one policy per thread (forward / backward pass)
    LaunchShape sf{}, sb{};   // forward / backward launch shapes
    StagedParams pf{}, pb{};
    size_t spill_bytes = 0;   // tiled spill: [tiles][rows of the backward program][backward tile]
};

// rows of one tile of the spill: the entries of the backward program (padded to whole stages for the lane kernel)
size_t spill_rows_of(const emo_graph *g, bool lane)
{
    return (size_t)(lane ? g->lbwd.steps_pad : g->bwd.steps) * g->bwd.lanes;
}

bool aligned16(const void *q) { return ((uintptr_t)q % 16) == 0; }

// Decides the plan for B policies (+ the virtual baseline column in the forward pass).
int make_plan(const emo_graph *g, int64_t B, bool want_base, bool need_bwd, const uint8_t *lvl, int64_t ldb,
              int64_t ldes_plain, int64_t ldo, uint32_t flags, PassPlan &pl)
{
    const int64_t big = (int64_t)1 << 28;
    const int64_t NBf = B + (want_base ? 1 : 0);
    const bool can_stage = !(flags & EMO_F_NO_STAGING) && ldb % 16 == 0 && aligned16(lvl) && ldb < big && ldes_plain < big && ldo < big;
    // One policy per thread gives twice the warps, which the path is short of; once a batch is so
    // large that even two policies per thread give every SM 16 consumer warps, the pair kernel is
    // the cheaper one (measured: 65 536 policies, 3 lanes: 0.96 ms against 1.02 ms for both passes,
    // 0.24 ms against 0.42 ms for the forward pass).
    const int64_t pair_warps = (NBf + 63) / 64 * std::max(g->fwd.lanes, g->bwd.lanes);
    const bool prefer_pair = (flags & EMO_F_PAIR_KERNEL) || (!(flags & EMO_F_LANE_KERNEL) && pair_warps >= 16 * (int64_t)g->sm_count);
    // Each pass picks its kernel (they only share the spill, whose tiling follows the backward pass).
    // A pass whose lane-kernel grid would need a second wave of blocks while the pair kernel's fits
    // the SMs once takes the pair kernel (a wide forward program: 18 lanes leave room for one group
    // of 32 policies per block; measured 2.7 ms against 4.5 ms).
    auto pick = [&](const Program &p, int rec_bytes, bool backward, int64_t NB, LaunchShape &ls, StagedParams &sp, bool &lane) {
        LaunchShape l1, l2;
        StagedParams s1, s2;
        const bool ok_lane = lane_shape(g, p, backward, NB, l1, s1);
        const bool ok_pair = staged_shape(g, p, rec_bytes, backward, NB, l2, s2);
        bool use_lane = ok_lane && !prefer_pair;
        if (use_lane && ok_pair && !(flags & EMO_F_LANE_KERNEL) && !backward && l1.grid > g->sm_count && l2.grid <= g->sm_count) use_lane = false;
        if (!use_lane && !ok_pair) use_lane = ok_lane;
        if (use_lane) { ls = l1; sp = s1; lane = true; return true; }
        if (ok_pair) { ls = l2; sp = s2; lane = false; return true; }
        return false;
    };
    pl.staged = can_stage && pick(g->fwd, g->dfwd.rec_bytes, false, NBf, pl.sf, pl.pf, pl.lane_f) &&
                (!need_bwd || pick(g->bwd, g->dbwd.rec_bytes, true, B, pl.sb, pl.pb, pl.lane_b));
    if (!pl.staged) {
        int rc = shape_for(g, g->fwd, NBf, pl.sf);
        if (rc == EMO_OK && need_bwd) rc = shape_for(g, g->bwd, B, pl.sb);
        return rc;
    }
    if (need_bwd) {
        const size_t tiles = ((size_t)B + pl.pb.ptile - 1) / pl.pb.ptile;
        pl.spill_bytes = tiles * spill_rows_of(g, pl.lane_b) * pl.pb.ptile * sizeof(int64_t);
    }
    return EMO_OK;
}

// One pass under a plan.  Forward: B policies from lvl plus, when base_T/base_E are given, the
// virtual all-max column.
int launch_pass(const emo_graph *g, const PassPlan &pl, bool backward, int64_t B, const uint8_t *lvl, int64_t ldb,
                int64_t *ES, int64_t ldes, int64_t *spill, int64_t *LS, int64_t *slack, int64_t ldo,
                int64_t *makespan, double *energy, int64_t *slack_sum, int32_t *n_critical,
                int64_t *base_T, double *base_E, int32_t *status, cudaStream_t st)
{
    const Program &p = backward ? g->bwd : g->fwd;
    const DevProgram &d = backward ? g->dbwd : g->dfwd;
    const int want_base = (!backward && (base_T || base_E)) ? 1 : 0;
    if (B + want_base == 0) return EMO_OK;
    const LaunchShape &s = backward ? pl.sb : pl.sf;
    PassParams a;
    a.rec = d.rec;
    a.rows = d.rows;
    a.rec_bytes = d.rec_bytes;
    a.steps = p.steps;
    a.lanes = p.lanes;
    a.Lp = p.Lp;
    a.L = g->h.L;
    a.slots = p.slots;
    a.sync = p.sync;
    a.groups = s.groups;
    a.want_base = want_base;
    a.B = B;
    a.lvl = lvl;
    a.ldb = ldb;
    a.ES = ES;
    a.ldes = ldes;
    a.spill = spill;
    a.spill_rows = (int64_t)spill_rows_of(g, pl.lane_b);
    a.spill_ptile = pl.staged ? pl.pb.ptile : 64;
    a.LS = LS;
    a.slack = slack;
    a.ldo = ldo;
    a.makespan = makespan;
    a.energy = energy;
    a.slack_sum = slack_sum;
    a.n_critical = n_critical;
    a.base_T = base_T;
    a.base_E = base_E;
    a.status = status;
    cudaEvent_t ev0 = g_pass_events[backward ? 2 : 0], ev1 = g_pass_events[backward ? 3 : 1];
    if (ev0) EMO_CUDA(cudaEventRecord(ev0, st));
    if (pl.staged) {
        StagedParams sp = backward ? pl.pb : pl.pf;
        sp.p = a;
        sp.vec_es = (ES && ldes % 2 == 0 && aligned16(ES)) ? 1 : 0;
        sp.vec_out = (ldo % 2 == 0 && aligned16(LS) && aligned16(slack)) ? 1 : 0;
        sp.want_sums = (slack_sum || n_critical) ? 1 : 0;
        // two register budgets: blocks of at most 512 threads may use 128 registers per thread
        // lean instantiation when the call asks for nothing beyond the spill (forward) or the slack
        // matrix with 16-byte aligned rows (backward); register budget by block size
        const bool extra = backward ? (LS != nullptr || sp.want_sums || !sp.vec_out) : (ES != nullptr);
        void (*kern)(StagedParams) = nullptr;
        if (backward ? pl.lane_b : pl.lane_f) {
            const DevProgramLane &di = backward ? g->lbwd : g->lfwd;
            LaneParams ip;
            const unsigned ne = (unsigned)sp.sc * (unsigned)p.lanes;
            sp.p.steps = di.steps_pad;
            sp.p.rows = di.rows;
            ip.tab_entry = di.tab_entry;
            ip.st.off_tab = ne * 32u;
            int nb = 0;
            auto bulk = [&](const void *src, unsigned per_entry, unsigned off, unsigned long long per_block) {
                sp.bsrc[nb] = (const unsigned char *)src;
                sp.bentry[nb] = per_entry;
                sp.boff[nb] = off;
                sp.bblock[nb] = per_block;
                ++nb;
            };
            bulk(di.ent, 32, 0, 0);
            bulk(di.tab, di.tab_entry, ip.st.off_tab, 0);
            if (backward) bulk(spill, (unsigned)sp.ptile * 8u, sp.off_es, (unsigned long long)a.spill_rows * sp.ptile * 8ull);
            sp.nbulk = nb;
            void (*kern_lane)(LaneParams) = nullptr;
            const bool extra_l = backward ? (LS != nullptr || sp.want_sums) : (ES != nullptr);
#define EMO_PICK_L(MAXT)                                                                                        \
    kern_lane = backward ? (extra_l ? emo_pass_lane<true, true, MAXT> : emo_pass_lane<true, false, MAXT>)           \
                        : (extra_l ? emo_pass_lane<false, true, MAXT> : emo_pass_lane<false, false, MAXT>)
            if (s.threads <= 512) EMO_PICK_L(512);
            else if (s.threads <= 768) EMO_PICK_L(768);
            else EMO_PICK_L(1024);
#undef EMO_PICK_L
            ip.sp = sp;
            EMO_CUDA(cudaFuncSetAttribute(kern_lane, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)g->smem_optin));      // the same value from every call
            kern_lane<<<s.grid, s.threads, s.smem, st>>>(ip);
        } else {
            sp.nbulk = 0;
            sp.bsrc[sp.nbulk] = d.rec; sp.bentry[sp.nbulk] = (unsigned)d.rec_bytes; sp.boff[sp.nbulk] = 0; sp.bblock[sp.nbulk] = 0;
            ++sp.nbulk;
            if (backward) {
                sp.bsrc[sp.nbulk] = (const unsigned char *)spill; sp.bentry[sp.nbulk] = (unsigned)sp.ptile * 8u; sp.boff[sp.nbulk] = sp.off_es;
                sp.bblock[sp.nbulk] = (unsigned long long)a.spill_rows * sp.ptile * 8ull;
                ++sp.nbulk;
            }
#define EMO_PICK(MAXT)                                                                                         \
    kern = backward ? (extra ? emo_pass_pair<true, true, MAXT> : emo_pass_pair<true, false, MAXT>)                 \
                    : (extra ? emo_pass_pair<false, true, MAXT> : emo_pass_pair<false, false, MAXT>)
        if (s.threads <= 512) EMO_PICK(512);
        else if (s.threads <= 768) EMO_PICK(768);
        else EMO_PICK(1024);
#undef EMO_PICK
        EMO_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)g->smem_optin));
        kern<<<s.grid, s.threads, s.smem, st>>>(sp);
        }
    } else if (backward) {
        if (s.smem > 48 * 1024) EMO_CUDA(cudaFuncSetAttribute(emo_pass_plain<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)g->smem_optin));
        emo_pass_plain<true><<<s.grid, s.threads, s.smem, st>>>(a);
    } else {
        if (s.smem > 48 * 1024) EMO_CUDA(cudaFuncSetAttribute(emo_pass_plain<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)g->smem_optin));
        emo_pass_plain<false><<<s.grid, s.threads, s.smem, st>>>(a);
    }
    EMO_CUDA(cudaGetLastError());
    if (ev1) EMO_CUDA(cudaEventRecord(ev1, st));
    return EMO_OK;
}


// ---- lane-stream program: upload, launch shape, launches -------------------------------------------
long long *g_flow_prof = nullptr;           // optional device array for the kernels' cycle counters (measurement hook)
long long g_wait_cycles = 4000000000LL;    // bound of every device-side wait of the 32-bit kernels (about two seconds)

int upload_flow(const Flow &f, DevFlow &d, bool intervals)
{
    if (!f.ok32 || f.stages == 0) return EMO_OK;
    const size_t per = (size_t)f.lanes * f.K;
    auto r16 = [](size_t x) { return (x + 15) / 16 * 16; };
    d.off_seg = (unsigned)r16((size_t)f.lanes * kHdrWords * 4);
    d.f_off_rec = (unsigned)r16(d.off_seg + (size_t)f.lanes * kSegBytes);
    d.f_off_pool = (unsigned)r16(d.f_off_rec + per * kFRecWords * 4);
    d.f_off_tab = (unsigned)r16(d.f_off_pool + (size_t)f.f.pool_stride * 4);
    d.blobF_bytes = (unsigned)r16(d.f_off_tab + per * f.Lp * 12);
    d.b_off_rec = d.f_off_rec;
    d.b_off_pool = (unsigned)r16(d.b_off_rec + per * kBRecWords * 4);
    d.b_off_lbes = (unsigned)r16(d.b_off_pool + (size_t)f.b.pool_stride * 4);
    d.b_off_tab = (unsigned)r16(d.b_off_lbes + per * 8);
    d.blobB_bytes = (unsigned)r16(d.b_off_tab + per * f.Lp * 4);
    std::vector<unsigned char> bf((size_t)f.stages * d.blobF_bytes, 0), bb((size_t)f.stages * d.blobB_bytes, 0);
    std::vector<uint32_t> pb((size_t)f.stages + 1);
    for (int st = 0; st <= f.stages; ++st) pb[st] = (uint32_t)f.push_base[st];
    for (int st = 0; st < f.stages; ++st) {
        d.max_push = std::max(d.max_push, (int)(pb[st + 1] - pb[st]));
        std::vector<uint32_t> hdr(f.hdr.begin() + (size_t)st * f.lanes * kHdrWords, f.hdr.begin() + (size_t)(st + 1) * f.lanes * kHdrWords);
        unsigned char *F = bf.data() + (size_t)st * d.blobF_bytes, *Bk = bb.data() + (size_t)st * d.blobB_bytes;
        std::memcpy(F, hdr.data(), hdr.size() * 4);
        std::memcpy(Bk, hdr.data(), hdr.size() * 4);
        std::memcpy(F + d.off_seg, &f.f.seg[(size_t)st * f.lanes * kSegBytes], (size_t)f.lanes * kSegBytes);
        std::memcpy(Bk + d.off_seg, &f.b.seg[(size_t)st * f.lanes * kSegBytes], (size_t)f.lanes * kSegBytes);
        std::memcpy(F + d.f_off_rec, &f.f.rec[(size_t)st * per * kFRecWords], per * kFRecWords * 4);
        std::memcpy(F + d.f_off_pool, &f.f.pool[(size_t)st * f.f.pool_stride], (size_t)f.f.pool_stride * 4);
        std::memcpy(F + d.f_off_tab, &f.tabF[(size_t)st * per * f.Lp * 3], per * f.Lp * 12);
        std::memcpy(Bk + d.b_off_rec, &f.b.rec[(size_t)st * per * kBRecWords], per * kBRecWords * 4);
        std::memcpy(Bk + d.b_off_pool, &f.b.pool[(size_t)st * f.b.pool_stride], (size_t)f.b.pool_stride * 4);
        std::memcpy(Bk + d.b_off_lbes, &f.lbes[(size_t)st * per], per * 8);
        std::memcpy(Bk + d.b_off_tab, &f.tabB[(size_t)st * per * f.Lp], per * f.Lp * 4);
    }
    int rc = upload(&d.blobF, bf.data(), bf.size());
    if (rc == EMO_OK) rc = upload(&d.blobB, bb.data(), bb.size());
    if (rc == EMO_OK && intervals) {
        d.f_off_meta = d.blobF_bytes;
        // per entry {lbES_v, group, dmin_v} and what tells whether the entry, or the run of plain entries that begins with it, ends inside
        // an interval: {earliest end of its last pack, that pack's group, shortest durations of all packs}; a run over several
        // groups (or 32 bits) names a group that no policy has and goes entry by entry.  One more entry is read behind the last.
        d.blobFI_bytes = (unsigned)r16(d.f_off_meta + (per + 1) * 32);
        std::vector<unsigned char> bi((size_t)f.stages * d.blobFI_bytes, 0);
        for (int st = 0; st < f.stages; ++st) {
            unsigned char *dst = bi.data() + (size_t)st * d.blobFI_bytes;
            std::memcpy(dst, bf.data() + (size_t)st * d.blobF_bytes, d.blobF_bytes);
            for (int ln = 0; ln < f.lanes; ++ln) {
                size_t e = (size_t)ln * f.K;
                auto check = [&](size_t first, size_t count) {
                    uint32_t grp = kNone;
                    uint64_t dsum = 0;
                    int64_t end = 0;
                    for (size_t j = first; j < first + count; ++j) {
                        const size_t q = (size_t)st * per + j;
                        const int64_t lb = f.lbes[q];
                        const uint32_t w[4] = {(uint32_t)(uint64_t)lb, (uint32_t)((uint64_t)lb >> 32), f.grp[q], f.dmin[q]};
                        std::memcpy(dst + d.f_off_meta + j * 32, w, 16);
                        if (f.grp[q] == kNone) continue;
                        grp = (grp == kNone || grp == f.grp[q]) ? f.grp[q] : kNone - 1u;
                        end = lb + (int64_t)f.dmin[q];
                        dsum += f.dmin[q];
                    }
                    if (dsum > 0xFFFFFFFFull) grp = kNone - 1u;
                    const uint32_t w[4] = {(uint32_t)(uint64_t)end, (uint32_t)((uint64_t)end >> 32), grp, (uint32_t)dsum};
                    std::memcpy(dst + d.f_off_meta + first * 32 + 16, w, 16);
                };
                const int nseg = (int)(f.hdr[((size_t)st * f.lanes + ln) * kHdrWords] & 255u);
                for (int i = 0; i < nseg; ++i) {
                    const uint32_t sg = f.f.seg[((size_t)st * f.lanes + ln) * kSegBytes + i];
                    if (sg & kSegSpecial) check(e++, 1);
                    if (sg & kSegRunMask) check(e, sg & kSegRunMask);
                    e += sg & kSegRunMask;
                }
            }
        }
        for (int ln = 0; ln < f.lanes; ++ln) {
            uint32_t last = kNone;
            for (int st = 0; st < f.stages; ++st)
                for (int k = 0; k < f.K; ++k) {
                    const uint32_t grp = f.grp[((size_t)st * f.lanes + ln) * f.K + k];
                    if (grp == kNone) continue;
                    d.packs++;
                    if (last != kNone && grp != last) d.switches++;
                    last = grp;
                }
        }
        rc = upload(&d.blobFI, bi.data(), bi.size());
    }
    if (rc == EMO_OK) rc = upload(&d.rows, f.rows.data(), f.rows.size() * 4);
    if (rc == EMO_OK) rc = upload(&d.push_base, pb.data(), pb.size() * 4);
    d.ready = rc == EMO_OK;
    return rc;
}

void free_flow(DevFlow &d)
{
    if (d.blobF) cudaFree(d.blobF);
    if (d.blobB) cudaFree(d.blobB);
    if (d.blobFI) cudaFree(d.blobFI);
    if (d.rows) cudaFree(d.rows);
    if (d.push_base) cudaFree(d.push_base);
    d = DevFlow();
}


// Look-up entries per chunk that the stages are cut for: enough to pay for the chunk's two waits, few enough that the
// look-up warps share a stage evenly (250 000 nodes, 55 look-up entries per stage: five chunks).
constexpr int kSpChunkTarget = 12;

// Lays the spine program out for the kernels.  A stage's look-up entries are the members of its segments that depend on
// the level (or carry energy), dealt to the chunks by length, longest segment first; the members of the other segments
// follow behind them (backward: they only store).  Backward the members of a segment lie last to first.  Sums are
// numbered compactly forward (segments whose sum is never read have none) and by segment backward.
int lay_out_spine(const Flow &f, DevSpine &d, SpineImage &im)
{
    const Spine &sp = f.spine;
    if (!f.ok32 || !sp.ok || f.stages == 0) return EMO_OK;
    auto r16 = [](size_t x) { return (x + 15) / 16 * 16; };
    const int stages = f.stages, lanes = f.lanes, K = f.K, Lp = f.Lp;
    struct StagePlan {
        std::vector<std::vector<uint32_t>> chunk;               // segments of every look-up chunk
        std::vector<int> fill;                                  // entries of every chunk, padded to a multiple of four
        std::vector<uint32_t> rest;                             // segments without look-ups
    };
    auto seg_word = [&](int st, uint32_t i, int k) { return sp.seg[((size_t)st * std::max(sp.max_segs, 1) + i) * kSpSegWords + k]; };
    auto seg_count = [&](int st, uint32_t i) { return (int)((seg_word(st, i, 0) >> 16) & 255u); };
    auto seg_flags = [&](int st, uint32_t i) { return seg_word(st, i, 0) >> 24; };
    int64_t active = 0;
    for (int st = 0; st < stages; ++st)
        for (uint32_t i = 0; i < sp.n_segs[st]; ++i)
            if (seg_flags(st, i) & (kSpSeg_PreF | kSpSeg_PreB)) active += seg_count(st, i);
    d.chunks = (int)std::max<int64_t>(1, std::min<int64_t>(kSpChunks - 1, (active + (int64_t)stages * kSpChunkTarget / 2) / ((int64_t)stages * kSpChunkTarget)));
    std::vector<StagePlan> plan((size_t)stages);
    int max_rest = 0;
    for (int st = 0; st < stages; ++st) {
        StagePlan &pl = plan[st];
        pl.chunk.resize((size_t)d.chunks);
        pl.fill.assign((size_t)d.chunks, 0);
        std::vector<uint32_t> act;
        int rest = 0;
        for (uint32_t i = 0; i < sp.n_segs[st]; ++i) {
            if (seg_flags(st, i) & (kSpSeg_PreF | kSpSeg_PreB)) act.push_back(i);
            else {
                pl.rest.push_back(i);
                rest += seg_count(st, i);
            }
        }
        std::stable_sort(act.begin(), act.end(), [&](uint32_t a, uint32_t b) { return seg_count(st, a) > seg_count(st, b); });
        for (uint32_t i : act) {
            const int c = (int)(std::min_element(pl.fill.begin(), pl.fill.end()) - pl.fill.begin());
            pl.chunk[c].push_back(i);
            pl.fill[c] += seg_count(st, i);
        }
        int total = 0;
        for (int &c : pl.fill) total += (c = (c + 3) / 4 * 4);
        d.nlook = std::max(d.nlook, total);
        max_rest = std::max(max_rest, (rest + 3) / 4 * 4);
    }
    if (d.nlook == 0) d.nlook = 4;
    const int nmem = d.nlook + max_rest;
    // forward words: one per operation that has a sum or whose value is pushed later, by the compiler's operation number.  A value
    // is pushed by the operation that produced it: the lane's last one before the node that asks for it.
    struct Push { uint32_t op, row; };
    std::vector<std::vector<Push>> push((size_t)stages);
    std::vector<std::vector<int>> word_op((size_t)stages);      // word of every forward operation (-1: none)
    std::vector<std::vector<int>> word_f((size_t)stages);       // ... by the compiler's word number
    size_t max_push_rec = 0;
    {
        std::vector<std::pair<int, uint32_t>> last((size_t)lanes, {-1, 0u});      // the lane's last operation
        for (int st = 0; st < stages; ++st)
            for (uint32_t i = 0; i < sp.f.n_ops[st]; ++i) {
                const uint32_t *w = &sp.f.ops[((size_t)st * sp.f.max_ops + i) * kSpOpWordsF];
                if (w[4] / 128u >= (uint32_t)lanes) continue;      // a merge or a filler
                auto &l = last[w[4] / 128u];
                // (a lane's first value needs no row: nothing lies in front of it)
                if ((w[7] & kSp_Push) && l.first >= 0) push[l.first].push_back({l.second, (uint32_t)sp.push_base[st] + ((w[7] >> 8) & 0xFFFu)});
                l = {st, i};
            }
        for (int st = 0; st < stages; ++st) {
            max_push_rec = std::max(max_push_rec, push[st].size());
            word_op[st].assign(sp.f.n_ops[st], -1);
            word_f[st].assign((size_t)sp.acc_words + 1, -1);
            int k = 0;
            for (uint32_t i = 0; i < sp.f.n_ops[st]; ++i) {
                const uint32_t *w = &sp.f.ops[((size_t)st * sp.f.max_ops + i) * kSpOpWordsF];
                if (!(w[7] & kSp_NoSum)) word_f[st][w[6] / 128u] = word_op[st][i] = k++;
            }
            for (const Push &q : push[st])
                if (word_op[st][q.op] < 0) word_op[st][q.op] = k++;
            d.f.words = std::max(d.f.words, k);
        }
    }
    d.f.zero = d.f.words;
    d.f.words += 2;
    d.b.zero = sp.max_segs;
    d.b.words = 2 * (sp.max_segs + 2);
    size_t max_term = 0;
    std::vector<size_t> n_term((size_t)stages, 0);
    for (int st = 0; st < stages; ++st) {
        for (uint32_t i = 0; i < sp.f.n_ops[st]; ++i) n_term[st] += (sp.f.ops[((size_t)st * sp.f.max_ops + i) * kSpOpWordsF + 7] & kSp_Terminal) != 0;
        max_term = std::max(max_term, n_term[st]);
    }
    d.f.off_pos = d.b.off_pos = 8 * kSpChunks;
    d.f.off_tab = (unsigned)r16(d.f.off_pos + (size_t)d.nlook * 4);
    d.f.w_bytes = (unsigned)r16(d.f.off_tab + (size_t)d.nlook * Lp * 12);
    d.b.off_mem = (unsigned)r16(d.b.off_pos + (size_t)d.nlook * 4);
    d.b.off_first = (unsigned)(d.b.off_mem + (size_t)nmem * 32);
    d.b.off_tab = (unsigned)r16(d.b.off_first + (size_t)(nmem + 31) / 32 * 4);
    d.b.w_bytes = (unsigned)r16(d.b.off_tab + (size_t)(d.nlook + 1) * Lp * 4);      // the last row stays zero: entries without look-ups
    const int NB = sp.bundle;
    const size_t op_bytes = kSpDevOpWords * 4, spare = (size_t)NB;      // a bundle behind the last is read ahead
    d.f.off_ops = (unsigned)(16 + max_term * 16);
    d.f.off_rec = (unsigned)(d.f.off_ops + (sp.f.max_ops + spare) * op_bytes);
    d.f.s_bytes = (unsigned)(d.f.off_rec + (max_push_rec + 3) / 4 * 32);
    d.b.off_ops = 16;
    d.b.off_rec = (unsigned)(d.b.off_ops + (sp.b.max_ops + spare) * op_bytes);
    // the completion walk: a stage's lanes are dealt to NB streams, the longest lane first (four records behind the last are
    // read ahead)
    std::vector<std::vector<std::vector<uint32_t>>> walk((size_t)stages);      // [stage][stream] segments, lane by lane, a lane's last to first
    size_t max_rounds = 0;
    for (int st = 0; st < stages; ++st) {
        std::vector<std::vector<uint32_t>> of((size_t)lanes);
        for (uint32_t i = 0; i < sp.n_segs[st]; ++i) of[seg_word(st, i, 0) & 255u].push_back(i);
        for (auto &l : of) std::sort(l.begin(), l.end(), [&](uint32_t x, uint32_t y) { return ((seg_word(st, x, 0) >> 8) & 255u) > ((seg_word(st, y, 0) >> 8) & 255u); });
        std::stable_sort(of.begin(), of.end(), [](const auto &x, const auto &y) { return x.size() > y.size(); });
        walk[st].resize((size_t)NB);
        for (auto &l : of) {
            auto &s0 = *std::min_element(walk[st].begin(), walk[st].end(), [](const auto &x, const auto &y) { return x.size() < y.size(); });
            s0.insert(s0.end(), l.begin(), l.end());
        }
        for (auto &w : walk[st]) max_rounds = std::max(max_rounds, (w.size() + 3) / 4 * 4);
    }
    d.b.s_bytes = (unsigned)(d.b.off_rec + (max_rounds + 4) * 16 * (size_t)NB);
    // all of it in one allocation and one copy (an allocation costs about a millisecond, more than a small graph's data)
    size_t total = 0;
    auto part = [&](size_t bytes) {
        const size_t at = total;
        total += round_up(bytes, 256);
        return at;
    };
    const size_t row_bytes = (size_t)stages * d.nlook * 4;
    im.at_fW = part((size_t)stages * d.f.w_bytes);
    im.at_fS = part((size_t)stages * d.f.s_bytes);
    im.at_bW = part((size_t)stages * d.b.w_bytes);
    im.at_bS = part((size_t)stages * d.b.s_bytes);
    im.at_rowsF = part(row_bytes);
    im.at_rowsB = part(row_bytes);
    im.at_pb = part(((size_t)stages + 1) * 4);
    std::vector<unsigned char> &host = im.host;
    host.assign(total, 0);
    uint32_t *rowsF = (uint32_t *)(host.data() + im.at_rowsF), *rowsB = (uint32_t *)(host.data() + im.at_rowsB), *pb = (uint32_t *)(host.data() + im.at_pb);
    std::fill(rowsF, rowsF + row_bytes / 4, kNone);
    std::fill(rowsB, rowsB + row_bytes / 4, kNone);
    for (int st = 0; st <= stages; ++st) pb[st] = (uint32_t)sp.push_base[st];
    const uint32_t unread = sp.unread_slot * 128u;
    size_t term0 = 0;
    for (int st = 0; st < stages; ++st) {
        d.max_push = std::max(d.max_push, (int)(pb[st + 1] - pb[st]));
        unsigned char *W = host.data() + im.at_fW + (size_t)st * d.f.w_bytes, *WB = host.data() + im.at_bW + (size_t)st * d.b.w_bytes;
        uint32_t *tableF = (uint32_t *)W, *tableB = (uint32_t *)WB, *posF = (uint32_t *)(W + d.f.off_pos), *posB = (uint32_t *)(WB + d.b.off_pos);
        uint32_t *mem = (uint32_t *)(WB + d.b.off_mem);
        for (int e = 0; e < nmem; ++e) {      // padding: no node, folded into the slot nobody reads
            mem[(size_t)e * 8] = kNone;
            mem[(size_t)e * 8 + 1] = unread;
        }
        uint32_t *first_bits = (uint32_t *)(WB + d.b.off_first);
        bool folds = false;
        auto put_seg = [&](uint32_t si, int &e, bool look) {
            const uint32_t w0 = seg_word(st, si, 0), wf = (uint32_t)std::max(word_f[st][seg_word(st, si, 1) / 128u], 0);
            const int ln = (int)(w0 & 255u), first = (int)((w0 >> 8) & 255u), cnt = seg_count(st, si);
            const bool sum = ((w0 >> 24) & kSpSeg_PreB) != 0;
            for (int j = 0; j < cnt; ++j, ++e) {
                const size_t qf = ((size_t)st * lanes + ln) * K + first + j, qb = ((size_t)st * lanes + ln) * K + first + cnt - 1 - j;
                const uint32_t *m = &sp.mem[qb * kSpMemWords];
                const uint32_t ends = (j == 0 ? kSpPos_First : 0u) | ((j == cnt - 1 && sum) ? kSpPos_Last : 0u);
                uint32_t *o = mem + (size_t)e * 8;
                std::memcpy(o, m, 32);
                o[3] = ends | (si << 16);
                folds = folds || m[1] != unread;
                if (j == 0) first_bits[e / 32] |= 1u << (e % 32);
                if (!look) continue;
                posB[e] = ends | (si << 16);
                posF[e] = ends | (wf << 16);
                rowsF[(size_t)st * d.nlook + e] = f.rows[qf];
                rowsB[(size_t)st * d.nlook + e] = f.rows[qb];
                std::memcpy(W + d.f.off_tab + (size_t)e * Lp * 12, &f.tabF[qf * Lp * 3], (size_t)Lp * 12);
                std::memcpy(WB + d.b.off_tab + (size_t)e * Lp * 4, &f.tabB[qb * Lp], (size_t)Lp * 4);
            }
        };
        // chunk table: first entry | entries << 16 (for the storing workers also: some entry is folded << 31)
        int e0 = 0;
        for (int c = 0; c < d.chunks; ++c) {
            int e = e0;
            folds = false;
            for (uint32_t si : plan[st].chunk[c]) put_seg(si, e, true);
            tableF[c] = tableB[c] = (uint32_t)e0 | ((uint32_t)plan[st].fill[c] << 16);
            tableB[kSpChunks + c] = tableB[c] | (folds ? 0x80000000u : 0u);
            e0 += plan[st].fill[c];
        }
        int er = d.nlook;
        folds = false;
        for (uint32_t si : plan[st].rest) put_seg(si, er, false);
        tableB[kSpChunks + d.chunks] = (uint32_t)d.nlook | ((uint32_t)((er - d.nlook + 3) / 4 * 4) << 16) | (folds ? 0x80000000u : 0u);

        uint32_t *hf = (uint32_t *)(host.data() + im.at_fS + (size_t)st * d.f.s_bytes), *hb = (uint32_t *)(host.data() + im.at_bS + (size_t)st * d.b.s_bytes);
        hf[0] = sp.f.n_ops[st] / (uint32_t)NB;
        hf[1] = (uint32_t)n_term[st];
        hf[2] = ((uint32_t)push[st].size() + 3u) / 4u * 4u;
        hb[0] = sp.b.n_ops[st] / (uint32_t)NB;
        for (auto &w : walk[st]) hb[2] = std::max(hb[2], (uint32_t)(w.size() + 3) / 4u * 4u);
        for (size_t t = 0; t < n_term[st]; ++t) {
            const uint64_t lb = sp.pool[(size_t)st * sp.max_pool + t];
            hf[4 + 4 * t + 0] = sp.term_slot[term0 + t] * 128u;
            hf[4 + 4 * t + 2] = (uint32_t)lb;
            hf[4 + 4 * t + 3] = (uint32_t)(lb >> 32);
        }
        term0 += n_term[st];
        auto put_op = [&](uint32_t *o, const uint32_t *w, uint32_t sum, uint32_t clear, uint32_t to) {
            const uint32_t v[kSpDevOpWords] = {w[0], w[2], sum * 128u, clear, w[1], w[3], w[4], w[5], to * 128u, 0u, 0u, 0u};
            std::memcpy(o, v, sizeof v);
        };
        // what lies behind the last operation is read ahead and must name words that exist: all zero
        for (uint32_t i = 0; i < sp.f.n_ops[st]; ++i) {
            const uint32_t *w = &sp.f.ops[((size_t)st * sp.f.max_ops + i) * kSpOpWordsF];
            const uint32_t sum = (w[7] & kSp_NoSum) ? (uint32_t)d.f.zero : (uint32_t)word_op[st][i];
            put_op((uint32_t *)((unsigned char *)hf + d.f.off_ops + i * op_bytes), w, sum, unread,
                   (uint32_t)(word_op[st][i] >= 0 ? word_op[st][i] : d.f.zero + 1));
        }
        {
            uint32_t *rec = (uint32_t *)((unsigned char *)hf + d.f.off_rec);
            for (uint32_t i = 0; i < hf[2]; ++i) {
                rec[2 * i] = i < push[st].size() ? (uint32_t)word_op[st][push[st][i].op] * 128u : 0u;
                rec[2 * i + 1] = i < push[st].size() ? push[st][i].row : kNone;
            }
        }
        std::vector<uint32_t> seg_of_word((size_t)sp.acc_words + 2, kNone), seg_flags_op((size_t)sp.max_segs + 1, 0);
        for (uint32_t i = 0; i < sp.n_segs[st]; ++i) seg_of_word[seg_word(st, i, 1) / 128u] = i;
        for (uint32_t i = 0; i < sp.b.n_ops[st]; ++i) {
            const uint32_t *w = &sp.b.ops[((size_t)st * sp.b.max_ops + i) * kSpOpWordsB];
            const uint32_t si = w[4] != unread ? seg_of_word[w[6] / 128u] : kNone;      // merge operations have no segment
            const bool sum = !(w[7] & kSp_NoSum);
            put_op((uint32_t *)((unsigned char *)hb + d.b.off_ops + i * op_bytes), w, sum ? si : (uint32_t)d.b.zero, w[8], si != kNone ? si : (uint32_t)d.b.zero + 1u);
            if (si != kNone) seg_flags_op[si] = ((w[7] & kSp_Push) ? kSpDev_Pop : 0u) | (sum ? 1u : 0u) | (w[7] & 0xFFFFFF00u);
        }
        uint32_t *rec = (uint32_t *)((unsigned char *)hb + d.b.off_rec);
        for (uint32_t i = 0; i < hb[2] + 4u; ++i)
            for (int k = 0; k < NB; ++k, rec += 4) {
                const std::vector<uint32_t> &w = walk[st][k];
                rec[0] = unread;
                rec[1] = (uint32_t)d.b.zero * 128u;
                rec[2] = (uint32_t)(d.b.zero + 1) * 128u;      // padding: words nobody reads
                if (i >= w.size()) continue;
                auto lane_of = [&](uint32_t j) { return seg_word(st, w[j], 0) & 255u; };
                const uint32_t ln = lane_of(i), fl = seg_flags_op[w[i]];
                rec[0] = ((uint32_t)(lanes + 2) + ln) * 128u;
                if (fl & 1u) rec[1] = w[i] * 128u;
                rec[2] = w[i] * 128u;
                rec[3] = (fl & ~1u) | ((i == 0 || lane_of(i - 1) != ln) ? kSpPos_First : 0u) | ((i + 1 == w.size() || lane_of(i + 1) != ln) ? kSpPos_Last : 0u);
            }
    }
    return EMO_OK;
}

// What launches take from a program: its sizes.  The tables are the compiler's and the layout's.
void keep_sizes(Flow &f)
{
    Flow k;
    k.ok32 = f.ok32;
    k.lanes = f.lanes;
    k.K = f.K;
    k.sync = f.sync;
    k.stages = f.stages;
    k.steps = f.steps;
    k.Lp = f.Lp;
    k.entries = f.entries;
    k.pushes = f.pushes;
    const Spine &s = f.spine;
    k.spine.ok = s.ok;
    k.spine.max_segs = s.max_segs;
    k.spine.max_pool = s.max_pool;
    k.spine.bundle = s.bundle;
    k.spine.acc_words = s.acc_words;
    k.spine.pushes = s.pushes;
    k.spine.segments = s.segments;
    k.spine.unread_slot = s.unread_slot;
    k.spine.f.slots = s.f.slots;
    k.spine.f.max_ops = s.f.max_ops;
    k.spine.b.slots = s.b.slots;
    k.spine.b.max_ops = s.b.max_ops;
    f = std::move(k);
}

int upload_spine(const SpineImage &im, DevSpine &d)
{
    if (im.host.empty()) return EMO_OK;
    const int rc = upload(&d.mem, im.host.data(), im.host.size());
    if (rc != EMO_OK) return rc;
    d.f.blobW = d.mem + im.at_fW;
    d.f.blobS = d.mem + im.at_fS;
    d.b.blobW = d.mem + im.at_bW;
    d.b.blobS = d.mem + im.at_bS;
    d.f.rows = (uint32_t *)(d.mem + im.at_rowsF);
    d.b.rows = (uint32_t *)(d.mem + im.at_rowsB);
    d.push_base = (uint32_t *)(d.mem + im.at_pb);
    d.ready = true;
    return EMO_OK;
}

void free_spine(DevSpine &d)
{
    if (d.mem) cudaFree(d.mem);
    d = DevSpine();
}

// Launch shape of the 32-bit kernels: both passes use the same policy tile (the restore list is laid
// out by tile), as many groups per block as cover the SMs once, two stage buffers (three when they fit).
struct FlowPlan {
    bool ok = false;
    int groups = 0, grid_f = 0, grid_b = 0, threads = 0;
    FlowParams pf, pb;
    size_t smem_f = 0, smem_b = 0;
    size_t restore_bytes = 0;
};

// intv: the plan of the forward kernel for time-interval policies (no level rows are staged; the blob carries
// 16 more bytes per entry; extra_fixed + G * extra_per_group bytes of the block are set aside for the change
// points and the block's columns of F).
bool flow_plan(const emo_graph *g, int64_t B, bool want_base, bool need_bwd, FlowPlan &pl, bool intv = false,
               size_t extra_fixed = 0, size_t extra_per_group = 0)
{
    const Flow &f = g->flow;
    const DevFlow &d = g->dflow;
    pl.ok = false;
    if (!f.ok32 || !d.ready || !g->smem_optin || f.stages == 0) return false;
    if (intv && !d.blobFI) return false;
    if (f.lanes * f.K > 32 * kFlowRowRegs) return false;
    const int64_t NBf = B + (want_base ? 1 : 0);
    const int64_t n_groups = (NBf + 31) / 32;
    const int gmax = std::min((32 - 2) / f.lanes, 15);
    if (gmax < 1) return false;
    const int64_t want = (n_groups + g->sm_count - 1) / g->sm_count;
    const size_t budget = g->smem_optin;
    for (int G = (int)std::max<int64_t>(1, std::min<int64_t>(gmax, want)); G >= 1; --G) {
        // four producer warps where the block has room for them (they share the level-row pieces)
        const int nprod = G * f.lanes + 4 <= 24 ? 4 : 2;
        const size_t P = 32 * (size_t)G;
        const size_t lvl_bytes = intv ? 0 : (size_t)G * f.lanes * f.K * 32;
        const size_t extra = intv ? round_up(extra_fixed + extra_per_group * G, 128) : 0;
        auto shape = [&](bool backward, FlowParams &p, size_t &smem) {
            const FlowDir &dir = backward ? f.b : f.f;
            const size_t slot_bytes = (size_t)dir.slots_tag * 256 + (size_t)dir.slots_set * 128;
            const size_t blob = backward ? d.blobB_bytes : (intv ? d.blobFI_bytes : d.blobF_bytes);
            const size_t rst = backward ? (size_t)d.max_push * P * 4 : 0;
            const size_t stage = round_up(blob + lvl_bytes + rst, 128);
            const size_t off_bar = round_up(G * slot_bytes, 16);
            const size_t head = round_up(off_bar + 256, 128) + extra;
            int nbuf = 0;
            for (int nb = 3; nb >= 2; --nb)
                if (head + nb * stage <= budget) { nbuf = nb; break; }
            if (!nbuf || nbuf * stage < (size_t)G * f.lanes * 32 * 16) return false;
            p = FlowParams();
            p.blob = backward ? d.blobB : (intv ? d.blobFI : d.blobF);
            p.rows = d.rows;
            p.push_base = d.push_base;
            p.blob_bytes = (unsigned)blob;
            p.off_seg = d.off_seg;
            p.off_rec = backward ? d.b_off_rec : d.f_off_rec;
            p.off_pool = backward ? d.b_off_pool : d.f_off_pool;
            p.off_tab = backward ? d.b_off_tab : d.f_off_tab;
            p.off_lbes = backward ? d.b_off_lbes : 0;
            p.off_meta = d.f_off_meta;
            p.off_brk = (unsigned)round_up(off_bar + 256, 128);
            p.off_Fs = p.off_brk + (unsigned)round_up(extra_fixed, 16);
            p.tab_row = (unsigned)f.Lp * (backward ? 4u : 12u);
            p.stages = f.stages;
            p.lanes = f.lanes;
            p.K = f.K;
            p.kshift = 0;
            while ((1 << p.kshift) < f.K) ++p.kshift;
            p.Lp = f.Lp;
            p.L = g->h.L;
            p.groups = G;
            p.ptile = (int)P;
            p.nbuf = nbuf;
            p.nprod = nprod;
            p.slot_bytes = (unsigned)slot_bytes;
            p.stage_bytes = (unsigned)stage;
            p.off_lvl = (unsigned)blob;
            p.off_rst = (unsigned)(blob + lvl_bytes);
            p.off_bar = (unsigned)off_bar;
            p.off_stage0 = (unsigned)head;
            p.pushes = f.pushes;
            p.restore_rows = f.pushes + f.lanes;
            p.wait_cycles = g_wait_cycles;
            p.stall_stage = -1;
            p.prof = nullptr;
            smem = head + nbuf * stage;
            return true;
        };
        if (!shape(false, pl.pf, pl.smem_f)) continue;
        if (need_bwd && !shape(true, pl.pb, pl.smem_b)) continue;
        pl.groups = G;
        pl.grid_f = (int)((n_groups + G - 1) / G);
        pl.grid_b = (int)(((B + 31) / 32 + G - 1) / G);
        pl.threads = (G * f.lanes + nprod) * 32;
        pl.restore_bytes = need_bwd ? round_up((size_t)pl.grid_f * (size_t)(f.pushes + f.lanes) * P * 4, 256) : 0;
        pl.ok = true;
        return true;
    }
    return false;
}

// Launches a kernel that may start before its predecessor in the stream ends (it waits for it where it needs it).  Measured:
// 400 nodes x 64, forward, backward and selection, 41 us one after the other, 31 ahead.
template <typename... A>
cudaError_t launch_ahead_grid(void (*kern)(A...), dim3 grid, int threads, size_t smem, cudaStream_t st, A... args)
{
    cudaLaunchConfig_t c = {};
    c.gridDim = grid;
    c.blockDim = dim3((unsigned)threads);
    c.dynamicSmemBytes = smem;
    c.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    c.attrs = attr;
    c.numAttrs = 1;
    return cudaLaunchKernelEx(&c, kern, args...);
}

template <typename... A>
cudaError_t launch_ahead(void (*kern)(A...), int grid, int threads, size_t smem, cudaStream_t st, A... args)
{
    return launch_ahead_grid(kern, dim3((unsigned)grid), threads, smem, st, args...);
}

// The opt-in shared-memory size is set once per kernel (not per launch: concurrent callers with
// different batch sizes would otherwise race on the attribute).
template <typename K>
int flow_optin(K kern, const emo_graph *g)
{
    return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)g->smem_optin) == cudaSuccess ? EMO_OK : EMO_E_CUDA;
}

int launch_flow_fwd(const emo_graph *g, const FlowPlan &pl, int64_t B, const uint8_t *lvl, int64_t ldb, uint32_t *restore,
                    int64_t *makespan, double *energy, int64_t *base_T, double *base_E, int32_t *status, uint32_t flags,
                    cudaStream_t st)
{
    FlowParams p = pl.pf;
    p.want_base = (base_T || base_E) ? 1 : 0;
    if (B + p.want_base == 0) return EMO_OK;
    p.B = B;
    p.lvl = lvl;
    p.ldb = ldb;
    p.restore = restore;
    p.makespan = makespan;
    p.energy = energy;
    p.base_T = base_T;
    p.base_E = base_E;
    p.status = status;
    p.prof = g_flow_prof;
    if (flags & EMO_F_TEST_STALL) p.stall_stage = p.stages / 2;
    cudaEvent_t ev0 = g_pass_events[0], ev1 = g_pass_events[1];
    if (ev0) EMO_CUDA(cudaEventRecord(ev0, st));
    void (*kern)(FlowParams) = nullptr;
    if (p.prof) kern = pl.threads <= 512 ? emo_flow_fwd<512, false, true> : (pl.threads <= 768 ? emo_flow_fwd<768, false, true> : emo_flow_fwd<1024, false, true>);
    else kern = pl.threads <= 512 ? emo_flow_fwd<512, false, false> : (pl.threads <= 768 ? emo_flow_fwd<768, false, false> : emo_flow_fwd<1024, false, false>);
    if (flow_optin(kern, g) != EMO_OK) { (void)cudaGetLastError(); return EMO_E_CUDA; }
    kern<<<pl.grid_f, pl.threads, pl.smem_f, st>>>(p);
    EMO_CUDA(cudaGetLastError());
    if (ev1) EMO_CUDA(cudaEventRecord(ev1, st));
    return EMO_OK;
}

int launch_flow_bwd(const emo_graph *g, const FlowPlan &pl, int64_t B, const uint8_t *lvl, int64_t ldb, uint32_t *restore,
                    int64_t *ES, int64_t *LS, int64_t *slack, int64_t ldo, int64_t *makespan, int64_t *slack_sum,
                    int32_t *n_critical, int32_t *status, uint32_t flags, cudaStream_t st)
{
    if (B == 0) return EMO_OK;
    FlowParams p = pl.pb;
    p.B = B;
    p.lvl = lvl;
    p.ldb = ldb;
    p.restore = restore;
    p.makespan = makespan;
    p.ES = ES;
    p.LS = LS;
    p.slack = slack;
    p.ldo = ldo;
    p.slack_sum = slack_sum;
    p.n_critical = n_critical;
    p.status = status;
    p.prof = g_flow_prof ? g_flow_prof + 131072 : nullptr;
    if (flags & EMO_F_TEST_STALL) p.stall_stage = p.stages / 2;
    cudaEvent_t ev0 = g_pass_events[2], ev1 = g_pass_events[3];
    if (ev0) EMO_CUDA(cudaEventRecord(ev0, st));
    const bool extra = ES || LS || slack_sum || n_critical;
    void (*kern)(FlowParams) = nullptr;
#define EMO_PICK_F(MAXT)                                                                                   \
    kern = p.prof ? (extra ? emo_flow_bwd<true, MAXT, true> : emo_flow_bwd<false, MAXT, true>)                 \
                  : (extra ? emo_flow_bwd<true, MAXT, false> : emo_flow_bwd<false, MAXT, false>)
    if (pl.threads <= 512) EMO_PICK_F(512);
    else if (pl.threads <= 768) EMO_PICK_F(768);
    else EMO_PICK_F(1024);
#undef EMO_PICK_F
    if (flow_optin(kern, g) != EMO_OK) { (void)cudaGetLastError(); return EMO_E_CUDA; }
    kern<<<pl.grid_b, pl.threads, pl.smem_b, st>>>(p);
    EMO_CUDA(cudaGetLastError());
    if (ev1) EMO_CUDA(cudaEventRecord(ev1, st));
    return EMO_OK;
}

// Launch shape of the spine kernels: a tile of 32 * G policies (kSpineTiles); two policies per spine thread up
// to three groups, else four (bundles of four, 8 threads per operation: always four, so that a row of 32 policies is one
// conflict-free access of those threads).
struct SpinePlan {
    bool ok = false, is_long = false;
    int groups = 0, vw = 1, vs = 1, grid_f = 0, grid_b = 0, threads_f = 0, threads_b = 0;
    const struct SpineKernels *k = nullptr;
    SpineParams pf, pb;
    size_t smem_f = 0, smem_b = 0;
    size_t restore_bytes = 0;
};

// The kernels of one shape.  The operations of a program come in bundles of its own size (the two programs of a graph are
// scheduled apart, so their lanes and with them their bundles may differ): a plan names the kernels of its program's.  SLACK,
// EXTRA: which backward kernels some tile below reaches.
struct SpineKernels {
    int vw, vs, nb, max_threads;
    void (*fwd)(SpineParams), (*bwd)(SpineParams), (*bwd_extra)(SpineParams);
};
template <int VW, int VS, int NB, int MAXT, bool SLACK, bool EXTRA>
constexpr SpineKernels spine_kernels()
{
    SpineKernels k = {VW, VS, NB, MAXT, emo_spine_fwd<VW, VS, NB, MAXT>, nullptr, nullptr};
    if constexpr (SLACK) k.bwd = emo_spine_bwd<VW, VS, NB, MAXT, false>;
    if constexpr (EXTRA) k.bwd_extra = emo_spine_bwd<VW, VS, NB, MAXT, true>;
    return k;
}
const SpineKernels kSpineKernels[] = {spine_kernels<1, 2, 2, 512, true, true>(), spine_kernels<1, 2, 2, 640, false, true>(), spine_kernels<2, 2, 2, 512, true, true>(),
                                      spine_kernels<2, 4, 2, 640, true, true>(), spine_kernels<4, 4, 2, 640, true, false>(), spine_kernels<1, 4, 4, 512, true, true>(),
                                      spine_kernels<2, 4, 4, 512, true, true>(), spine_kernels<2, 4, 4, 640, false, true>(), spine_kernels<4, 4, 4, 640, true, false>()};

// Tiles of policies: groups of 32 per block, policies per worker and (bundles of two) per spine thread, what a wave of blocks
// costs (in units of a group); whether wide graphs have it, and calls without and with per-node ES / LS or sums.  A batch takes
// the tile whose waves cost least.
// Measured (both passes, ms).  All outputs: four policies per worker leave a storing warp one entry at a time, fewer are faster:
// 10 000 nodes x 14 000 policies 1.15 with three groups, 1.79 with four at four per worker; x 18 900 1.33 with four at two per
// worker, 1.82 at four; 500 nodes x 19 000 0.108 with six, 0.185 at four per worker; the one loss met is 25 000 nodes x
// 37 000, 5.98 against 5.87.  Slack alone: six groups where eight would leave half of the SMs without a block, 1 013 nodes x 19 000 0.160 / 0.187;
// but four rather than three, 25 000 x 9 600 1.54 / 1.73.  The cost of six: 500 nodes x 60 000 take 0.224 in four waves of four
// and 0.238 in three of six.
struct SpineTile {
    int groups, vw, vs;
    double cost;
    bool wide, slack, extra;
};
constexpr SpineTile kSpineTiles[] = {{8, 4, 4, 10.0, false, true, false}, {8, 2, 4, 10.0, false, false, true}, {6, 2, 4, 8.1, false, true, true},
                                     {4, 4, 4, 6.0, true, true, false}, {4, 2, 4, 6.0, true, false, true}, {3, 1, 2, 5.0, false, false, true},
                                     {2, 2, 2, 4.0, true, true, true}, {1, 1, 2, 3.0, true, true, true}};

// What a launch shape depends on beside the program and the batch.
struct SpineChip {
    int sm_count;
    size_t smem;
};

bool spine_plan_for(const emo_graph *g, const SpineChip &chip, const Flow &f, const DevSpine &d, int64_t B, bool want_base, bool need_bwd, bool extra, SpinePlan &pl)
{
    const Spine &sp = f.spine;
    pl.ok = false;
    if (!f.ok32 || !sp.ok || !d.ready || !chip.smem || f.stages == 0) return false;
    const int64_t NBf = B + (want_base ? 1 : 0);
    const int64_t n_groups = (NBf + 31) / 32;
    const size_t budget = chip.smem;
    const bool wide = sp.bundle > 2;
    double best = 0.0;
    for (const SpineTile &tile : kSpineTiles) {
        if ((wide && !tile.wide) || (extra ? !tile.extra : !tile.slack)) continue;
        const int64_t blocks = (n_groups + tile.groups - 1) / tile.groups;
        const double cost = (double)((blocks + chip.sm_count - 1) / chip.sm_count) * tile.cost;
        if (pl.ok && cost >= best) continue;
        SpinePlan cand;
        const int G = tile.groups;
        const size_t P = 32 * (size_t)G;
        const int VW = tile.vw, VS = wide ? 4 : tile.vs, spines = (int)P / (32 / sp.bundle * VS), subs = G / VW;
        auto shape = [&](bool backward, SpineParams &p, size_t &smem, int &threads) {
            const SpineDir &dir = backward ? sp.b : sp.f;
            const DevSpineDir &dd = backward ? d.b : d.f;
            // warps: 16 (128 registers per thread) up to two policy groups, else 20 (96).  What the spine (backward also the
            // completion walk) and the producers leave goes to the workers, backward two fifths of it to the look-ups (250 000
            // nodes x 16 384 policies: 5 look-up and 9 storing warps); multiples of the sub-tiles.
            const int avail = (G <= 2 ? 16 : 20) - (backward ? 2 : 1) * spines - 2;
            const int pushers = !backward && need_bwd ? subs : 0;
            const int look = (backward ? std::max(avail * 2 / 5, subs) : std::min(avail - pushers, 12)) / subs * subs;
            const int posts = backward ? (avail - look) / subs * subs : pushers;
            const size_t acc = (size_t)dd.words * P * 4, slots = (size_t)dir.slots * P * 4;
            const size_t rst = backward ? (size_t)d.max_push * P * 4 : 0;
            const size_t wbuf = round_up((size_t)dd.w_bytes + (size_t)d.nlook * P, 128), sbuf = round_up(dd.s_bytes + rst, 128);
            const size_t off_bar = round_up(slots, 128), off_rows = round_up(off_bar + kSpBarBytes, 16);
            const size_t rowbuf = round_up((size_t)d.nlook * 4 + 512, 16), off_w0 = round_up(off_rows + kSpRowRing * rowbuf, 128);      // (up to 128 row numbers are read past the last)
            // buffers: the look-up warps run up to nacc stages ahead of the spine and, backward, the storing warps one behind it
            static const int kTry[8][3] = {{6, 4, 3}, {5, 4, 3}, {4, 3, 3}, {4, 2, 3}, {3, 2, 3}, {4, 2, 2}, {3, 2, 2}, {2, 2, 2}};      // {nw, ns, nacc}
            for (auto &t : kTry) {
                // no worker may skip more stages than there are buffers of sums (a barrier's parity tells two phases apart)
                const int n_look = std::min(look / subs, d.chunks * t[2]) * subs, n_post = backward ? std::min(posts / subs, (d.chunks + 1) * t[2]) * subs : posts;
                // (the warps' partial results at the end take the place of the stage buffers)
                const size_t total = off_w0 + std::max(t[0] * wbuf + t[1] * sbuf + t[2] * acc, (size_t)std::max(n_look * 8, n_post * 16) * 32 * VW);
                if (total > budget) continue;
                p = SpineParams();
                p.blobW = dd.blobW;
                p.blobS = dd.blobS;
                p.rows = dd.rows;
                p.push_base = d.push_base;
                p.w_bytes = dd.w_bytes;
                p.s_bytes = dd.s_bytes;
                p.off_pos = dd.off_pos;
                p.off_mem = dd.off_mem;
                p.off_first = dd.off_first;
                p.off_tab = dd.off_tab;
                p.tab_row = (unsigned)f.Lp * (backward ? 4u : 12u);
                p.off_ops = dd.off_ops;
                p.nlook = d.nlook;
                p.chunks = d.chunks;
                p.chunks_post = d.chunks + 1;
                p.stages = f.stages;
                p.lanes = f.lanes;
                p.Lp = f.Lp;
                p.L = g->h.L;
                p.groups = G;
                p.ptile = (int)P;
                p.workers = n_look;
                p.posts = n_post;
                p.nw = t[0];
                p.ns = t[1];
                p.nacc = t[2];
                p.wbuf_bytes = (unsigned)wbuf;
                p.sbuf_bytes = (unsigned)sbuf;
                p.acc_bytes = (unsigned)acc;
                p.slot_bytes = (unsigned)slots;
                p.off_lvl = dd.w_bytes;
                p.off_rst = dd.s_bytes;
                p.off_bar = (unsigned)off_bar;
                p.off_rows = (unsigned)off_rows;
                p.rowbuf_bytes = (unsigned)rowbuf;
                p.off_w0 = (unsigned)off_w0;
                p.off_s0 = p.off_w0 + (unsigned)(t[0] * wbuf);
                p.off_acc0 = p.off_s0 + (unsigned)(t[1] * sbuf);
                p.off_rec = dd.off_rec;
                p.zero_word = (unsigned)dd.zero;
                p.comp_off = (unsigned)(sp.max_segs + 2) * 128u;
                p.c_slot0 = f.lanes + 2;
                p.pushes = sp.pushes;
                p.restore_rows = sp.pushes + f.lanes;
                p.wait_cycles = g_wait_cycles;
                p.stall_stage = -1;
                smem = total;
                threads = ((backward ? 2 : 1) * spines + n_look + n_post + 2) * 32;
                return true;
            }
            return false;
        };
        if (!shape(false, cand.pf, cand.smem_f, cand.threads_f)) continue;
        if (need_bwd && !shape(true, cand.pb, cand.smem_b, cand.threads_b)) continue;
        for (const SpineKernels &k : kSpineKernels)
            if (!cand.k && k.vw == VW && k.vs == VS && k.nb == sp.bundle && cand.threads_f <= k.max_threads && (!need_bwd || cand.threads_b <= k.max_threads) &&
                (extra ? k.bwd_extra : k.bwd))
                cand.k = &k;
        if (!cand.k) continue;
        cand.groups = G;
        cand.vw = VW;
        cand.vs = VS;
        cand.grid_f = (int)blocks;
        cand.grid_b = (int)(((B + 31) / 32 + G - 1) / G);
        cand.restore_bytes = need_bwd ? round_up((size_t)cand.grid_f * (size_t)(sp.pushes + f.lanes) * P * 4, 256) : 0;
        cand.ok = true;
        best = cost;
        pl = cand;
    }
    return pl.ok;
}

// Up to two policy groups per SM a block has shared memory to spare and its stages are bound by latency: the program with the
// longer stages.  Measured (both passes, ms, long / short stages): 10 000 nodes x 4 096 policies 0.60 / 0.77, x 9 000 0.69 / 0.86;
// 25 000 x 2 000 0.78 / 0.83, x 8 192 1.03 / 1.07; 1 013 x 4 096 0.085 / 0.096.  Above that the larger buffers cost tiles or stages in
// flight: 1 013 x 65 536 0.50 / 0.36.  On wide graphs only up to one group: 18 lanes, 51 000 x 1 000 1.82 / 2.09, x 8 192 2.7 / 2.49.
bool spine_plan_on(const emo_graph *g, const SpineChip &chip, int64_t B, bool want_base, bool need_bwd, bool extra, SpinePlan &pl)
{
    const int64_t n_groups = (B + (want_base ? 1 : 0) + 31) / 32;
    if (n_groups <= (g->lflow.lanes > 8 ? 1 : 2) * (int64_t)chip.sm_count && spine_plan_for(g, chip, g->lflow, g->dlong, B, want_base, need_bwd, extra, pl)) {
        pl.is_long = true;
        return true;
    }
    return spine_plan_for(g, chip, g->sflow, g->dspine, B, want_base, need_bwd, extra, pl);
}

// extra: the call asks for ES, LS or the sums
bool spine_plan(const emo_graph *g, int64_t B, bool want_base, bool need_bwd, bool extra, SpinePlan &pl)
{
    return spine_plan_on(g, SpineChip{g->sm_count, g->smem_optin}, B, want_base, need_bwd, extra, pl);
}

int launch_spine_fwd(const emo_graph *g, const SpinePlan &pl, int64_t B, const uint8_t *lvl, int64_t ldb, uint32_t *restore,
                     int64_t *makespan, double *energy, int64_t *base_T, double *base_E, int32_t *status, uint32_t flags,
                     cudaStream_t st)
{
    SpineParams p = pl.pf;
    p.want_base = (base_T || base_E) ? 1 : 0;
    if (B + p.want_base == 0) return EMO_OK;
    p.B = B;
    p.lvl = lvl;
    p.ldb = ldb;
    p.restore = restore;
    p.makespan = makespan;
    p.energy = energy;
    p.base_T = base_T;
    p.base_E = base_E;
    p.status = status;
    p.prof = g_flow_prof;
    if (flags & EMO_F_TEST_STALL) p.stall_stage = p.stages / 2;
    cudaEvent_t ev0 = g_pass_events[0], ev1 = g_pass_events[1];
    if (ev0) EMO_CUDA(cudaEventRecord(ev0, st));
    void (*kern)(SpineParams) = pl.k->fwd;
    if (flow_optin(kern, g) != EMO_OK) { (void)cudaGetLastError(); return EMO_E_CUDA; }
    EMO_CUDA(launch_ahead(kern, pl.grid_f, pl.threads_f, pl.smem_f, st, p));
    if (ev1) EMO_CUDA(cudaEventRecord(ev1, st));
    return EMO_OK;
}

int launch_spine_bwd(const emo_graph *g, const SpinePlan &pl, int64_t B, const uint8_t *lvl, int64_t ldb, uint32_t *restore,
                     int64_t *ES, int64_t *LS, int64_t *slack, int64_t ldo, int64_t *makespan, int64_t *slack_sum,
                     int32_t *n_critical, int32_t *status, uint32_t flags, cudaStream_t st)
{
    if (B == 0) return EMO_OK;
    SpineParams p = pl.pb;
    p.B = B;
    p.lvl = lvl;
    p.ldb = ldb;
    p.restore = restore;
    p.makespan = makespan;
    p.ES = ES;
    p.LS = LS;
    p.slack = slack;
    p.ldo = ldo;
    auto out_aligned = [&](const void *q) { return ((uintptr_t)q % (8u * (unsigned)pl.vw)) == 0; };
    p.vec_out = ldo % pl.vw == 0 && out_aligned(ES) && out_aligned(LS) && out_aligned(slack);
    p.slack_sum = slack_sum;
    p.n_critical = n_critical;
    p.status = status;
    p.prof = g_flow_prof ? g_flow_prof + 131072 : nullptr;
    if (flags & EMO_F_TEST_STALL) p.stall_stage = p.stages / 2;
    cudaEvent_t ev0 = g_pass_events[2], ev1 = g_pass_events[3];
    if (ev0) EMO_CUDA(cudaEventRecord(ev0, st));
    const bool extra = ES || LS || slack_sum || n_critical;
    void (*kern)(SpineParams) = extra ? pl.k->bwd_extra : pl.k->bwd;
    if (flow_optin(kern, g) != EMO_OK) { (void)cudaGetLastError(); return EMO_E_CUDA; }
    EMO_CUDA(launch_ahead(kern, pl.grid_b, pl.threads_b, pl.smem_b, st, p));
    if (ev1) EMO_CUDA(cudaEventRecord(ev1, st));
    return EMO_OK;
}

// Whether a call takes the spine kernels: the program exists and either the caller asks for them (EMO_F_SPINE_KERNEL) or
// they are the faster ones.
bool spine_allowed(const emo_graph *g, int64_t B, const uint8_t *lvl, int64_t ldb, int64_t ldo, uint32_t flags)
{
    const int64_t big = (int64_t)1 << 28;
    if (!g->sflow.ok32 || !g->sflow.spine.ok || !g->dspine.ready) return false;
    if (flags & (EMO_F_NO_STAGING | EMO_F_PAIR_KERNEL | EMO_F_LANE_KERNEL | EMO_F_FLOW_KERNEL)) return false;
    // Measured (both passes, ms, spine / the best of the others): 1 013 nodes x 65 536 policies 0.36 / 0.90; 10 000 x 4 096
    // 0.77 / 2.30; 75 000 x 10 001 forward 1.28 / 1.89; 250 000 x 16 384 15.0 / 20.4.  On wide graphs one warp carries the
    // recurrence of all lanes: 18 lanes, 128 039 nodes x 8 192 policies (two groups per SM) 6.2 / 9.05; 51 000 x 333 to
    // 4 500 (one group) 2.09 / 2.05 and 6 400 nodes 0.31 / 0.30 with stages of four positions, so there the others stay; with the
    // program of longer stages 1.82 and 0.25.
    if (!(flags & EMO_F_SPINE_KERNEL)) {
        const int64_t per_sm = ((B + 1 + 31) / 32 + g->sm_count - 1) / std::max(g->sm_count, 1);
        if (g->sflow.lanes > 8 && per_sm < 2 && !g->dlong.ready) return false;
    }
    return ldb % 16 == 0 && aligned16(lvl) && ldb < big && ldo < big;
}

// The contracted graph for a call without outputs per node, unless the caller names its kernels.
const emo_graph *joined_for(const emo_graph *g, uint32_t flags)
{
    return flags & (EMO_F_NO_STAGING | EMO_F_PAIR_KERNEL | EMO_F_LANE_KERNEL | EMO_F_FLOW_KERNEL | EMO_F_SPINE_KERNEL | EMO_F_TEST_STALL) ? nullptr : g->joined;
}

// Whether a call takes the 32-bit lane-stream kernels: the program exists, the level matrix can be
// fetched in 16-byte pieces, and either the caller asks for them (EMO_F_FLOW_KERNEL) or the batch is
// large (for the graph or for the SMs).  Measured on the five workloads: on the 250 000-node graph with 16 384 policies they are
// the faster pair (25.8 ms against 30.1 ms for both passes) and need 1.6 GB of workspace instead of
// 37.7 GB; on the smaller workloads, where a block holds one or two policy groups and every step is
// latency, the 64-bit staged kernels with their one-step-ahead fetch are faster (2.3 ms against 3.7 ms on
// 10 000 nodes x 4 096 policies).
bool flow_allowed(const emo_graph *g, int64_t B, const uint8_t *lvl, int64_t ldb, int64_t ldo, uint32_t flags)
{
    const int64_t big = (int64_t)1 << 28;
    if (!g->flow.ok32 || !g->dflow.ready) return false;
    if (flags & (EMO_F_NO_STAGING | EMO_F_PAIR_KERNEL | EMO_F_LANE_KERNEL)) return false;
    if (!(flags & EMO_F_FLOW_KERNEL)) {
        // large batches, and on narrow graphs every batch with more than three policy groups per SM (where the spine
        // kernels stop; 75 000 nodes x 16 384 policies: 6.8 ms against 9.0 ms for the 64-bit staged kernels)
        const int64_t per_sm = ((B + 1 + 31) / 32 + g->sm_count - 1) / std::max(g->sm_count, 1);
        if ((int64_t)g->h.n * B < ((int64_t)1 << 31) && !(g->flow.lanes <= 8 && per_sm > 3)) return false;
    }
    return ldb % 16 == 0 && aligned16(lvl) && ldb < big && ldo < big;
}

// ---- slices -------------------------------------------------------------------------------------------------
// What a launch needs to know of a slice program.
void size_slices(const Slices &s, DevSlice &d)
{
    d = DevSlice();
    for (int k = 0; k < s.count; ++k) {
        SliceHdr h;
        std::memcpy(&h, s.blob.data() + s.off[(size_t)k], sizeof(h));
        d.words = std::max(d.words, h.words);
        d.head = std::max(d.head, h.head);
        d.nodes = std::max(d.nodes, h.nodes);
        for (int i = 0; i < 2; ++i) {
            d.len[i] = std::max(d.len[i], h.dir[i].len);
            d.steps[i] = std::max(d.steps[i], h.dir[i].steps);
            d.slots1[i] = std::max(d.slots1[i], h.dir[i].slots1);
            d.slots2[i] = std::max(d.slots2[i], h.dir[i].slots2);
        }
    }
    d.count = s.count;
    d.cols = s.cols;
    d.Lp = s.Lp;
    d.group = s.group;
    d.groups = s.groups;
    d.ready = s.ok;
}

int upload_slices(const Slices &s, DevSlice &d)
{
    std::vector<uint4> index((size_t)s.count);
    for (int k = 0; k < s.count; ++k) {
        SliceHdr h;
        std::memcpy(&h, s.blob.data() + s.off[(size_t)k], sizeof(h));
        index[(size_t)k] = make_uint4(s.off[(size_t)k], h.nodes, h.node0, std::min(h.head, 0xFFFFu) | std::min(h.words, 0xFFFFu) << 16);
    }
    const void *src[5] = {s.blob.data(), index.data(), s.rec.data(), s.tabT.data(), s.tabE.data()};
    const size_t bytes[5] = {s.blob.size() * 4, index.size() * sizeof(uint4), s.rec.size() * 4, s.tabT.size() * 4, s.tabE.size() * 8};
    size_t at[5], total = 0;
    for (int i = 0; i < 5; ++i) {
        at[i] = total;
        total += round_up(bytes[i], 256);
    }
    unsigned char *mem = nullptr;
    cudaError_t rc = cudaMalloc(&mem, total);
    for (int i = 0; i < 5 && rc == cudaSuccess; ++i) rc = cudaMemcpy(mem + at[i], src[i], bytes[i], cudaMemcpyHostToDevice);
    if (rc != cudaSuccess) {
        (void)cudaGetLastError();
        if (mem) cudaFree(mem);
        d = DevSlice();
        return rc == cudaErrorMemoryAllocation ? EMO_E_OOM : EMO_E_CUDA;
    }
    d.mem = mem;
    d.blob = (uint32_t *)(d.mem + at[0]);
    d.index = (uint4 *)(d.mem + at[1]);
    d.rec = (uint4 *)(d.mem + at[2]);
    d.tabT = (uint32_t *)(d.mem + at[3]);
    d.tabE = (double *)(d.mem + at[4]);
    return EMO_OK;
}

// How a call takes the slice kernels.
struct SlicePlan {
    int shape = 0;                  // index into kSliceP
    SliceParams p, pv;              // of the matrices' kernel and the chaining, of the values' kernel; workspace pointers as offsets
    size_t smem_m = 0, smem_v = 0, smem_g = 0, smem_s = 0, ws = 0;
    int whole = -1;                 // index into kSliceWhole: one block per policy does everything (p, smem_m)
};
struct SliceKernels {
    void (*matrix)(SliceParams), (*values)(SliceParams), (*single)(SliceParams);
    int threads;
};
template <int SHAPE, int NT>
constexpr SliceKernels slice_kernels()
{
    return {emo_slice_matrix<kSliceP[SHAPE], kSliceS[SHAPE], NT>, emo_slice_values<kSliceP[SHAPE], kSliceS[SHAPE], NT, false>, emo_slice_values<kSliceP[SHAPE], 1, NT, true>, NT};
}
const SliceKernels kSliceKernels[kSliceShapes] = {slice_kernels<0, 256>(), slice_kernels<1, 256>(), slice_kernels<2, 256>()};

// The kernels that chain matrices: threads per unit and block, buffers of the ring.  Matrices of more than 16 columns are not
// multiplied (the product of two costs as many additions as a chaining of all slices), their slices are chained one by one.
struct SliceChain {
    int cols, lanes, threads, ring;
    void (*group)(SliceParams), (*scan)(SliceParams);
};
template <int LPP, int D, int CW>
constexpr SliceChain slice_chain_of()
{
    return {CW, LPP, 32, D, emo_slice_group<LPP, D, CW>, emo_slice_scan<LPP, D, CW>};
}
const SliceChain kSliceChains[] = {slice_chain_of<8, 16, 4>(), slice_chain_of<8, 16, 8>(), slice_chain_of<16, 8, 12>(), slice_chain_of<16, 8, 16>(),
                                   {emo::kSliceMaxCols, 256, 256, 6, nullptr, emo_slice_scan_wide<6>}};
const SliceChain &slice_chain(int cols)
{
    int i = 0;
    while (kSliceChains[i].cols < cols) ++i;
    return kSliceChains[i];
}

// One block per policy: most slices, threads.
struct SliceWhole {
    int slices, threads;
    void (*kern)(SliceParams);
};
const SliceWhole kSliceWhole[] = {{4, 512, emo_slice_whole<4, 512>}, {8, 512, emo_slice_whole<8, 512>}};

bool slice_plan(const emo_graph *g, int64_t B, bool want_base, bool need_bwd, int shape, SlicePlan &pl)
{
    const DevSlice &d = g->dslice;
    if (!d.ready) return false;
    if (d.head > 0xFFFF) return false;
    const int64_t nb = B + (want_base ? 1 : 0), P = kSliceP[shape];
    const int64_t tiles = (nb + P - 1) / P;
    pl.shape = shape;
    SliceParams &p = pl.p;
    p = SliceParams();
    p.blob = d.blob;
    p.index = d.index;
    p.rec = d.rec;
    p.tabT = d.tabT;
    p.tabE = d.tabE;
    p.count = d.count;
    p.cols = d.cols;
    p.Lp = d.Lp;
    p.L = g->h.L;
    p.dirs = need_bwd ? 2 : 1;
    const SliceChain &ch = slice_chain(d.cols);
    const bool grouped = d.groups > 1 && ch.group;
    p.group = grouped ? d.group : d.count;
    p.groups = grouped ? d.groups : 1;
    p.B = B;
    p.nb = nb;
    p.nbp = tiles * P;
    if (tiles * d.count > 0x7FFFFFFF || (int64_t)p.groups * p.nbp > 0x7FFFFFFF) return false;
    p.tiles = (int)tiles;
    // workspace: matrices, groups' matrices, values that enter, energies
    size_t at = 0;
    auto take = [&](size_t bytes) {
        const size_t here = at;
        at += round_up(bytes, 256);
        return (unsigned char *)nullptr + here;
    };
    const size_t size = (size_t)d.cols * d.cols;
    if (d.count > 1) {
        for (int i = 0; i < p.dirs; ++i) {
            p.mat[i] = (int32_t *)take((size_t)d.count * p.nbp * size * 4);
            p.gmat[i] = (int32_t *)take(p.groups > 1 ? (size_t)p.groups * p.nbp * size * 4 : 0);
            p.state[i] = (long long *)take((size_t)d.count * p.nbp * d.cols * 8);
        }
        p.epart = (double *)take((size_t)d.count * p.nbp * 8);
        p.gepart = (double *)take((size_t)p.groups * p.nbp * 8);
    }
    pl.ws = at;
    // shared memory
    pl.pv = p;
    const int NT = kSliceKernels[shape].threads, S = d.count > 1 ? kSliceS[shape] : 1;
    auto layout = [&](SliceParams &q, const unsigned (&slots)[2], unsigned slot_bytes) {
        size_t o = round_up((size_t)d.head * 4, 128);
        q.at_rec = (unsigned)o;
        o += (size_t)d.nodes * 16;
        for (int i = 0; i < q.dirs; ++i) {
            q.at_ops[i] = (unsigned)o;
            o += (size_t)(d.steps[i] + 1) * 32;
        }
        for (int i = 0; i < q.dirs; ++i) {
            o = round_up(o, 128);
            q.at_inc[i] = (unsigned)o;
            o += (size_t)d.len[i] * P * 4;
        }
        for (int i = 0; i < q.dirs; ++i) {
            o = round_up(o, 128);
            q.at_slot[i] = (unsigned)o;
            o += (size_t)slots[i] * slot_bytes;
        }
        o = round_up(o, 128) + (S > 1 ? 32 : 0);      // (slices side by side in a warp: not on the same banks)
        q.slice_bytes = (unsigned)o;
        q.at_red = (unsigned)(o * S);
        return o * S + (size_t)NT * 8 + (size_t)P * 8;
    };
    pl.smem_m = layout(pl.p, d.slots1, 4u * (unsigned)P * (unsigned)d.cols);
    pl.smem_v = layout(pl.pv, d.slots2, 8u * (unsigned)P);
    pl.whole = -1;
    if (shape == 0 && d.count > 1 && d.cols <= 32 && d.words <= 0xFFFF && nb <= 0x7FFFFFFF) {
        for (int w = 0; w < 2 && pl.whole < 0; ++w) {
            const SliceWhole &k = kSliceWhole[w];
            if (d.count > k.slices) continue;
            SliceParams q = p;
            size_t o = (size_t)d.words * 4;
            q.at_rec = (unsigned)o;
            o += (size_t)d.nodes * 16;
            for (int i = 0; i < q.dirs; ++i) {
                q.at_inc[i] = (unsigned)o;
                o += round_up((size_t)d.len[i] * 4, 16);
            }
            for (int i = 0; i < q.dirs; ++i) {
                q.at_slot[i] = (unsigned)o;
                o += round_up(std::max((size_t)d.slots1[i] * d.cols * 4, (size_t)d.slots2[i] * 8), 16);
            }
            o = round_up(o, 128) + 32;      // (slices side by side in a warp: not on the same banks)
            q.slice_bytes = (unsigned)o;
            q.at_red = (unsigned)(o * d.count);
            const size_t total = o * d.count + (size_t)k.threads * 8 + 16 + (size_t)2 * k.slices * d.cols * 8 + (size_t)2 * k.slices * size * 4;
            if (total > g->smem_optin) continue;
            pl.p = q;
            pl.smem_m = total;
            pl.ws = 0;
            pl.whole = w;
        }
    }
    if (pl.whole >= 0) return true;
    pl.smem_g = (size_t)(ch.threads / ch.lanes) * size * 4 * ch.ring;
    pl.smem_s = pl.smem_g + (size_t)(ch.threads / ch.lanes) * d.cols * 16;
    const size_t budget = g->smem_optin;
    return (d.count == 1 || pl.smem_m <= budget) && pl.smem_v <= budget && pl.smem_g <= budget && pl.smem_s <= budget;
}

// Most policies (the all-max one included) of a call that the slice kernels take.  Their time grows with the policies, that of the
// spine kernels not before they fill the SMs.  Measured (us, slices / the others):
//   slack       10 000 nodes x 257 105 / 593, x 1 025 348 / 596; 25 000 x 1 025 676 / 770, x 1 501 964 / 768; 1 013 x 1 025 55 / 76, x 1 501 71 / 76
//   all outputs 10 000 x 1 501 532 / 689; 25 000 x 1 025 712 / 911, x 1 501 1 013 / 911
//   forward     10 000 x 1 025 98 / 263; 25 000 x 1 501 250 / 249; 400 x 1 501 16 / 14
//   one slice   213 x 4 097 20.7 / 23.3 (forward 12.0 / 12.9, both the call)
//   12 columns  10 000 x 769 slack 209 / 290, all outputs 229 / 361, forward 84 / 117, x 1 025 271 / 291, 293 / 362, 105 / 118; 50 000 x 769 961 / 1 380
//   16 columns  10 000 x 513 slack 201 / 283, all outputs 218 / 362, forward 84 / 102, x 769 286 / 282, 303 / 362, 113 / 103
//   20 columns  50 000 x 65 slack 500 / 1 355, forward 318 / 476, x 129 793 / 1 356, 540 / 476; 12 014 x 129 slack 293 / 477
//   36 columns  24 014 x 33 slack 423 / 793, x 65 616 / 791
//   40 columns  12 839 (18 lanes): slack x 17 192 / 447, x 65 438 / 447; forward x 17 109 / 123, x 65 207 / 123
// (Up to 16 columns slices are chained in groups; wider ones one by one, and a policy's matrices go with the columns' square.)
int64_t slice_limit(const emo_graph *g, bool need_bwd, bool extra)
{
    const DevSlice &d = g->dslice;
    if (d.count == 1) return 4352;
    if (d.cols <= 8) return need_bwd ? (extra ? 1300 : 1100) : 1400;
    if (d.cols <= 16) return d.cols <= 12 ? 900 : 600;
    return 65536 / ((int64_t)d.cols * d.cols) / (need_bwd ? 1 : 2);
}

// Call flags that name other kernels.
constexpr uint32_t kNotSlices = EMO_F_NO_STAGING | EMO_F_PAIR_KERNEL | EMO_F_LANE_KERNEL | EMO_F_FLOW_KERNEL | EMO_F_SPINE_KERNEL | EMO_F_TEST_STALL;

// Blocks of a call on the slice kernels.  Measured (us): one block per policy where all are there at once, 400 nodes x 64 16.6 / 21.5,
// 1 013 x 64 23.7 / 26.3 in three kernels.  Else one policy per block (four slices) for up to four, and for wide matrices, which fill
// a warp's lanes with one policy (12 839 nodes x 16, 40 columns 192 / 293); 16 policies instead of 8 where a block's columns are the
// work, forward (250 000 x 256 440 / 603), or where three large blocks still fit an SM and there are plenty (250 000 x 256 1 749 /
// 2 002; but 10 000 x 257 115 / 105, two blocks and a half).
bool slice_shape(const emo_graph *g, int64_t B, bool want_base, bool need_bwd, uint32_t flags, SlicePlan &pl)
{
    const DevSlice &d = g->dslice;
    const int64_t nb = B + (want_base ? 1 : 0);
    const bool one = slice_plan(g, B, want_base, need_bwd, 0, pl);
    // forward on two to four slices: one block per policy and SM, else the spine kernel's one launch (400 nodes x 1 025 14.2 against 18.8)
    if (!need_bwd && d.count > 1 && d.count <= 4 && !(flags & EMO_F_SLICE_KERNEL) && !(one && pl.whole >= 0 && nb <= g->sm_count)) return false;
    const int64_t at_once = one ? (int64_t)g->sm_count * std::min<int64_t>(4, (int64_t)g->smem_optin / (int64_t)std::max<size_t>(pl.whole >= 0 ? pl.smem_m : pl.smem_v, 1)) : 0;
    if (one && (d.count == 1 ? nb <= at_once : (pl.whole >= 0 ? nb <= at_once : nb <= 4 || d.cols > 16))) return true;
    if (d.count > 1 && nb > 32 && slice_plan(g, B, want_base, need_bwd, 2, pl) &&
        (!need_bwd || (3 * pl.smem_v <= (size_t)200 * 1024 && (int64_t)d.count * pl.p.tiles >= 9 * (int64_t)g->sm_count)))
        return true;
    return slice_plan(g, B, want_base, need_bwd, 1, pl);
}

// Whether a call takes the slice kernels, and with which blocks (a workspace for all policies at once provided).
bool slice_allowed(const emo_graph *g, int64_t B, bool want_base, bool need_bwd, bool extra, uint32_t flags, SlicePlan &pl)
{
    if (!g->dslice.ready || (flags & kNotSlices)) return false;
    const int64_t nb = B + (want_base ? 1 : 0);
    if (nb == 0) return false;
    if (!(flags & EMO_F_SLICE_KERNEL) && nb > slice_limit(g, need_bwd, extra)) return false;
    return slice_shape(g, B, want_base, need_bwd, flags, pl);
}

// ---- workspace of the slice kernels
// Matrices and entering values of every slice take 0.5 MB a policy and direction on 250 000 nodes.  Forward calls need next to
// nothing otherwise, so they would ask for 0.76 GB there with 1 399 policies: beyond kSliceWs a call runs in tiles of policies, one
// after the other.  Measured (us, 250 000 nodes x 1 024, one tile / 512 / 256 / 128 / 64 a tile): forward 1 605 / 1 666 / 1 783 / 1 973 /
// 2 406, slack 6 498 / 6 657 / 6 861 / 7 144 / 7 688 (slack calls have room for one tile: the other kernels' restore lists need more).
constexpr size_t kSliceWs = (size_t)256 << 20;
constexpr int64_t kSliceLeastTile = 64;          // fewer policies a tile (unless the call has no more) are left to the other kernels

size_t slice_policy_bytes(const emo_graph *g, bool need_bwd)
{
    const DevSlice &d = g->dslice;
    if (d.count <= 1) return 0;
    const size_t size = (size_t)d.cols * d.cols * 4, groups = d.groups > 1 ? (size_t)d.groups : 0;
    return (need_bwd ? 2 : 1) * (((size_t)d.count + groups) * size + (size_t)d.count * d.cols * 8) + ((size_t)d.count + std::max<size_t>(groups, 1)) * 8;
}

// ... of nb policies; no plan of as many needs more (blocks of up to 16 policies, eight arrays in pieces of 256 bytes).
size_t slice_ws(const emo_graph *g, int64_t nb, bool need_bwd)
{
    return slice_policy_bytes(g, need_bwd) * round_up((size_t)nb, 16) + 8 * 256;
}

// What a call on B policies asks for; it suffices for every smaller call too.
size_t slice_call_ws(const emo_graph *g, int64_t B, bool need_bwd, uint32_t flags)
{
    const DevSlice &d = g->dslice;
    if (!d.ready || d.count <= 1 || (flags & kNotSlices)) return 0;
    const int64_t nb = flags & EMO_F_SLICE_KERNEL ? B + 1 : std::min(B + 1, slice_limit(g, need_bwd, true));
    SlicePlan pl;
    if (nb <= 0 || !slice_plan(g, 1, false, need_bwd, 1, pl)) return 0;
    return std::min(slice_ws(g, nb, need_bwd), std::max(kSliceWs, slice_ws(g, kSliceLeastTile + 16, need_bwd)));
}

// Bytes that the slice kernels may use of a caller's workspace, behind its head.  They move it 16 bytes at a time: none where it is not
// aligned to that (forward calls do not touch it otherwise, so there it may lie anywhere).
size_t slice_room(const void *ws, size_t ws_bytes, size_t head)
{
    return ws && aligned16(ws) && ws_bytes > head ? ws_bytes - head : 0;
}

// What a call reads and writes.
struct SliceCall {
    const uint8_t *lvl;
    int64_t ldb;
    int64_t *ES, *LS, *slack;
    int64_t ldo;
    int64_t *makespan;
    double *energy;
    int64_t *slack_sum;
    int32_t *n_critical;
    int64_t *base_T;
    double *base_E;
};

// One tile of a call: policies b0 and following, on a plan of its own (its pointers are set here).  first, last: of the call (its events).
int launch_slices(const emo_graph *g, SlicePlan &pl, const SliceCall &c, int64_t b0, bool first, bool last, unsigned char *ws, cudaStream_t st)
{
    const SliceKernels &k = kSliceKernels[pl.shape];
    auto from = [&](auto *x) { return x ? x + b0 : x; };
    for (SliceParams *p : {&pl.p, &pl.pv}) {
        p->lvl = from(c.lvl);
        p->ldb = c.ldb;
        p->ES = from(c.ES);
        p->LS = from(c.LS);
        p->slack = from(c.slack);
        p->ldo = c.ldo;
        p->makespan = from(c.makespan);
        p->energy = from(c.energy);
        p->slack_sum = from(c.slack_sum);
        p->n_critical = from(c.n_critical);
        p->base_T = c.base_T;
        p->base_E = c.base_E;
        for (int i = 0; i < p->dirs; ++i) {
            p->mat[i] = (int32_t *)(ws + (size_t)p->mat[i]);
            p->gmat[i] = (int32_t *)(ws + (size_t)p->gmat[i]);
            p->state[i] = (long long *)(ws + (size_t)p->state[i]);
        }
        p->epart = (double *)(ws + (size_t)p->epart);
        p->gepart = (double *)(ws + (size_t)p->gepart);
    }
    const SliceParams &p = pl.p;
    const int slices = p.count > 1 ? kSliceS[pl.shape] : 1, blocks = (p.count + slices - 1) / slices * p.tiles;
    // both passes run side by side: the backward events enclose the kernel that writes the outputs where it is one of its own
    const bool back = last && pl.p.dirs > 1;
    cudaEvent_t ev0 = first ? g_pass_events[0] : nullptr, ev1 = last ? g_pass_events[1] : nullptr, ev2 = back ? g_pass_events[2] : nullptr, ev3 = back ? g_pass_events[3] : nullptr;
    if (ev0) EMO_CUDA(cudaEventRecord(ev0, st));
    if (pl.whole >= 0) {
        const SliceWhole &w = kSliceWhole[pl.whole];
        if (flow_optin(w.kern, g) != EMO_OK) { (void)cudaGetLastError(); return EMO_E_CUDA; }
        EMO_CUDA(launch_ahead(w.kern, (int)p.nb, w.threads, pl.smem_m, st, p));
        for (cudaEvent_t ev : {ev1, ev2, ev3})
            if (ev) EMO_CUDA(cudaEventRecord(ev, st));
        return EMO_OK;
    }
    if (p.count > 1) {
        if (flow_optin(k.matrix, g) != EMO_OK) { (void)cudaGetLastError(); return EMO_E_CUDA; }
        EMO_CUDA(launch_ahead(k.matrix, blocks, k.threads, pl.smem_m, st, p));
        const SliceChain &ch = slice_chain(p.cols);
        const int64_t units = (int64_t)p.groups * p.nbp, per = ch.threads / ch.lanes;
        const dim3 grid((unsigned)((units + per - 1) / per), (unsigned)p.dirs);
        if (p.groups > 1) {
            if (flow_optin(ch.group, g) != EMO_OK) { (void)cudaGetLastError(); return EMO_E_CUDA; }
            EMO_CUDA(launch_ahead_grid(ch.group, grid, ch.threads, pl.smem_g, st, p));
        }
        if (flow_optin(ch.scan, g) != EMO_OK) { (void)cudaGetLastError(); return EMO_E_CUDA; }
        EMO_CUDA(launch_ahead_grid(ch.scan, grid, ch.threads, pl.smem_s, st, p));
    }
    if (p.count > 1)
        for (cudaEvent_t ev : {ev1, ev2})
            if (ev) EMO_CUDA(cudaEventRecord(ev, st));
    if (p.count == 1 || p.dirs > 1) {
        void (*values)(SliceParams) = p.count == 1 ? k.single : k.values;
        if (flow_optin(values, g) != EMO_OK) { (void)cudaGetLastError(); return EMO_E_CUDA; }
        EMO_CUDA(launch_ahead(values, blocks, k.threads, pl.smem_v, st, pl.pv));
    }
    for (cudaEvent_t ev : {p.count == 1 ? ev1 : nullptr, p.count == 1 ? ev2 : nullptr, ev3})
        if (ev) EMO_CUDA(cudaEventRecord(ev, st));
    return EMO_OK;
}

// A call in tiles of as many policies as the workspace holds; false where too few of them fit.
bool slice_tiles(const emo_graph *g, int64_t B, bool need_bwd, uint32_t flags, const SliceCall &c, unsigned char *area, size_t room, cudaStream_t st, int &rc)
{
    const bool base = c.base_T || c.base_E;      // (the last tile has the all-max policy too)
    int64_t tile = std::min<int64_t>(B, (int64_t)(room / std::max<size_t>(slice_policy_bytes(g, need_bwd), 1))) / 16 * 16 - 16;
    while (tile >= kSliceLeastTile && slice_ws(g, tile + 1, need_bwd) > room) tile -= 16;
    if (tile < kSliceLeastTile) return false;
    const int64_t tiles = (B + tile - 1) / tile, rest = B - (tiles - 1) * tile;
    SlicePlan each, end;
    if (!slice_shape(g, tile, false, need_bwd, flags, each) || !slice_shape(g, rest, base, need_bwd, flags, end) || each.ws > room || end.ws > room) return false;
    rc = EMO_OK;
    for (int64_t k = 0; k < tiles && rc == EMO_OK; ++k) {
        SlicePlan pl = k + 1 < tiles ? each : end;
        rc = launch_slices(g, pl, c, k * tile, k == 0, k + 1 == tiles, area, st);
    }
    return true;
}

// Runs a call on the slice kernels; false where it does not take them.
bool slice_call(const emo_graph *g, int64_t B, bool need_bwd, uint32_t flags, const SliceCall &c, void *ws, size_t ws_bytes, size_t head, cudaStream_t st, int &rc)
{
    SlicePlan pl;
    if (!slice_allowed(g, B, c.base_T || c.base_E, need_bwd, c.ES || c.LS || c.slack_sum || c.n_critical, flags, pl)) return false;
    const size_t room = slice_room(ws, ws_bytes, head);
    unsigned char *const area = room ? (unsigned char *)ws + head : nullptr;
    if (pl.ws > room) return slice_tiles(g, B, need_bwd, flags, c, area, room, st, rc);
    rc = launch_slices(g, pl, c, 0, true, true, area, st);
    return true;
}

int launch_validate(const emo_graph *g, int64_t B, const uint8_t *lvl, int64_t ldb, int32_t *status, cudaStream_t st)
{
    if (!status) return EMO_E_INVALID_ARG;
    int64_t total = (int64_t)g->h.rows * B;
    if (total == 0) return EMO_OK;
    int grid = (int)std::min<int64_t>((total + 255) / 256, (int64_t)g->sm_count * 16);
    emo_validate_levels<<<grid, 256, 0, st>>>(lvl, ldb, g->h.rows, B, g->h.L, status);
    EMO_CUDA(cudaGetLastError());
    return EMO_OK;
}

}  // namespace

extern "C" {

const char *emo_strerror(int code)
{
    switch (code) {
        case EMO_OK: return "ok";
        case EMO_E_INVALID_ARG: return "invalid argument";
        case EMO_E_NOT_TOPOLOGICAL: return "nodes are not numbered topologically";
        case EMO_E_RANGE: return "value out of the supported range";
        case EMO_E_OVERFLOW: return "slowest-level makespan does not fit below 2^62 ns";
        case EMO_E_NONFINITE: return "non-finite energy";
        case EMO_E_OOM: return "out of memory or workspace too small";
        case EMO_E_CUDA: return "CUDA runtime error";
        case EMO_E_TIMEOUT: return "bounded device wait ran out";
        case EMO_E_UNSUPPORTED: return "no path for these arguments (see the call's description)";
        default: return "unknown status";
    }
}

int emo_set_pass_events(void *fwd_start, void *fwd_stop, void *bwd_start, void *bwd_stop)
{
    g_pass_events[0] = (cudaEvent_t)fwd_start;
    g_pass_events[1] = (cudaEvent_t)fwd_stop;
    g_pass_events[2] = (cudaEvent_t)bwd_start;
    g_pass_events[3] = (cudaEvent_t)bwd_stop;
    return EMO_OK;
}

int emo_call_path(const emo_graph *g, int64_t B, const uint8_t *lvl, int64_t ldb, int64_t ldo, int need_slack, uint32_t flags)
{
    if (!g || B < 0) return EMO_E_INVALID_ARG;
    if (g->host_only) return EMO_E_CUDA;
    if (g->generic) return 3;
    for (const emo_graph *e : {need_slack ? nullptr : joined_for(g, flags), g}) {
        SpinePlan sp;
        if (e && spine_allowed(e, B, lvl, ldb, need_slack ? ldo : 0, flags) && spine_plan(e, B, true, need_slack != 0, false, sp)) return sp.vw == 1 ? 4 : 5;
    }
    if (flow_allowed(g, B, lvl, ldb, need_slack ? ldo : 0, flags)) {
        FlowPlan fp;
        if (flow_plan(g, B, true, need_slack != 0, fp)) return 2;
    }
    PassPlan pl;
    const int64_t ld_ws = (int64_t)round_up((size_t)B, 16);
    int rc = make_plan(g, B, true, need_slack != 0, lvl, ldb, ld_ws, ldo, flags, pl);
    if (rc) return rc;
    return pl.staged ? 1 : 0;
}

int emo_graph_contracted(const emo_graph *g, int32_t *nodes)
{
    if (!g || !nodes) return EMO_E_INVALID_ARG;
    *nodes = g->joined ? g->joined->h.n : 0;
    return EMO_OK;
}

int emo_call_slices(const emo_graph *g, int64_t B, int need_slack, uint32_t flags)
{
    if (!g || B < 0) return EMO_E_INVALID_ARG;
    if (g->host_only) return EMO_E_CUDA;
    SlicePlan cp;
    for (const emo_graph *e : {need_slack ? nullptr : joined_for(g, flags), g}) {
        if (!e) continue;
        if (slice_allowed(e, B, true, need_slack != 0, false, flags, cp)) return e->dslice.count;
        if (e != g && e->dspine.ready) return 0;
    }
    return 0;
}

int emo_measure_int_issue(double *ops_per_s, void *scratch_dev, void *stream)
{
    if (!ops_per_s || !scratch_dev) return EMO_E_INVALID_ARG;
    int dev = 0, sms = 0;
    EMO_CUDA(cudaGetDevice(&dev));
    EMO_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    cudaStream_t st = (cudaStream_t)stream;
    cudaEvent_t e0, e1;
    EMO_CUDA(cudaEventCreate(&e0));
    EMO_CUDA(cudaEventCreate(&e1));
    const int grid = sms * 8, iters = 2048;                    // 64 warps per SM, 8 chains x 4 x iters operations per thread
    unsigned long long *sink = (unsigned long long *)scratch_dev;
    int rc = EMO_OK;
    for (int op = 0; op < 4 && rc == EMO_OK; ++op) {
        float best = 0.f;
        for (int rep = 0; rep < 4; ++rep) {                    // the first repetition warms up
            cudaEventRecord(e0, st);
            if (op == 0) emo_int_chains<0><<<grid, 256, 0, st>>>(sink, iters, 12345u);
            else if (op == 1) emo_int_chains<1><<<grid, 256, 0, st>>>(sink, iters, 12345u);
            else if (op == 2) emo_int_chains<2><<<grid, 256, 0, st>>>(sink, iters, 12345u);
            else emo_int_chains<3><<<grid, 256, 0, st>>>(sink, iters, 12345u);
            cudaEventRecord(e1, st);
            if (cudaEventSynchronize(e1) != cudaSuccess || cudaGetLastError() != cudaSuccess) { rc = EMO_E_CUDA; break; }
            float ms = 0.f;
            cudaEventElapsedTime(&ms, e0, e1);
            if (rep > 0 && (best == 0.f || ms < best)) best = ms;
        }
        const double warp_ops = (double)grid * 8.0 /* warps per block */ * 8.0 * 4.0 * iters;
        ops_per_s[op] = best > 0.f ? warp_ops / (best * 1e-3) : 0.0;
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    return rc;
}

int emo_measure_warp_costs(double *cycles, void *scratch_dev, void *stream)
{
    if (!cycles || !scratch_dev) return EMO_E_INVALID_ARG;
    cudaStream_t st = (cudaStream_t)stream;
    long long *out = (long long *)scratch_dev;                 // 9 results, then one zero word the kernel reads
    const int iters = 512;
    if (cudaMemsetAsync(scratch_dev, 0, 128, st) != cudaSuccess) return EMO_E_CUDA;
    long long h[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    for (int rep = 0; rep < 2; ++rep) {                        // the first repetition warms up
        emo_warp_costs<<<1, 160, 0, st>>>(out, (const unsigned *)(out + 12), iters, 12345u);
        if (cudaMemcpyAsync(h, out, sizeof(h), cudaMemcpyDeviceToHost, st) != cudaSuccess) return EMO_E_CUDA;
        if (cudaStreamSynchronize(st) != cudaSuccess || cudaGetLastError() != cudaSuccess) return EMO_E_CUDA;
    }
    for (int k = 0; k < 8; ++k) cycles[k] = (double)h[k] / iters;
    return EMO_OK;
}

int emo_set_flow_counters(void *dev)
{
    g_flow_prof = (long long *)dev;
    return EMO_OK;
}

int emo_set_wait_limit(int64_t cycles)
{
    if (cycles <= 0) return EMO_E_INVALID_ARG;
    g_wait_cycles = cycles;
    return EMO_OK;
}

static size_t pass_ws_bytes(const emo_graph *g, int64_t B, int need_slack, uint32_t flags, int aligned);

static int32_t hop_depth(const HostGraph &h)
{
    std::vector<int32_t> hop((size_t)std::max(h.n, 1), 0);
    int32_t depth = 0;
    for (int32_t v = 0; v < h.n; ++v) {
        int32_t a = 0;
        for (int64_t e = h.row_ptr[v]; e < h.row_ptr[v + 1]; ++e) a = std::max(a, hop[h.col[e]] + 1);
        hop[v] = a;
        depth = std::max(depth, a + 1);
    }
    return depth;
}

// inner: this is a contracted graph; only what its calls read is compiled (the spine and slice programs).
static int load_graph(int32_t n, const int64_t *row_ptr, const int32_t *col, const int32_t *level_ptr,
                      int32_t n_levels, int32_t L, const int64_t *lat, const double *energy,
                      const int32_t *group_of, uint32_t flags, bool inner, emo_graph **out)
{
    if (!out) return EMO_E_INVALID_ARG;
    *out = nullptr;
    if (n < 0 || !row_ptr) return EMO_E_INVALID_ARG;
    if (L < 1 || L > 255) return EMO_E_RANGE;
    if (n > 0 && (!lat || !energy)) return EMO_E_INVALID_ARG;
    if (row_ptr[0] != 0) return EMO_E_INVALID_ARG;
    for (int32_t v = 0; v < n; ++v)
        if (row_ptr[v + 1] < row_ptr[v]) return EMO_E_INVALID_ARG;
    const int64_t m = row_ptr[n];
    if (m > 0 && !col) return EMO_E_INVALID_ARG;
    int32_t max_span = 0;
    for (int32_t v = 0; v < n; ++v)
        for (int64_t e = row_ptr[v]; e < row_ptr[v + 1]; ++e) {
            if (col[e] < 0 || col[e] >= n) return EMO_E_INVALID_ARG;
            if (col[e] >= v) return EMO_E_NOT_TOPOLOGICAL;
            max_span = std::max(max_span, v - col[e]);
        }
    if (level_ptr) {
        // the whole array is checked before anything is indexed with it
        if (n_levels < 0 || level_ptr[0] != 0 || level_ptr[n_levels] != n) return EMO_E_INVALID_ARG;
        for (int32_t l = 0; l < n_levels; ++l)
            if (level_ptr[l] < 0 || level_ptr[l + 1] > n || level_ptr[l + 1] < level_ptr[l]) return EMO_E_INVALID_ARG;
        try {
            std::vector<int32_t> lev((size_t)std::max(n, 1));
            for (int32_t l = 0; l < n_levels; ++l)
                for (int32_t v = level_ptr[l]; v < level_ptr[l + 1]; ++v) lev[v] = l;
            for (int32_t v = 0; v < n; ++v)
                for (int64_t e = row_ptr[v]; e < row_ptr[v + 1]; ++e)
                    if (lev[col[e]] >= lev[v]) return EMO_E_NOT_TOPOLOGICAL;
        } catch (const std::bad_alloc &) {
            return EMO_E_OOM;
        }
    }
    for (int64_t i = 0; i < (int64_t)n * L; ++i) {
        if (lat[i] < 0 || lat[i] >= ((int64_t)1 << 32)) return EMO_E_RANGE;
        if (!std::isfinite(energy[i])) return EMO_E_NONFINITE;
    }
    int32_t rows = n;
    if (group_of) {
        rows = 0;
        for (int32_t v = 0; v < n; ++v) {
            if (group_of[v] < -1) return EMO_E_INVALID_ARG;
            rows = std::max(rows, group_of[v] + 1);
        }
    }

    // (declared before the threads below, so that however the load ends it waits for them before the graph goes)
    struct Owned {
        emo_graph *g = nullptr;
        ~Owned() { emo_graph_free(g); }
    } owned, joined;
    emo_graph *const g = owned.g = new (std::nothrow) emo_graph();
    if (!g) return EMO_E_OOM;
    g->host_only = (flags & EMO_F_HOST_ONLY) != 0;
    Slices slices;
    try {
        HostGraph &h = g->h;
        h.n = n;
        h.L = L;
        h.rows = rows;
        h.m = m;
        h.max_span = max_span;
        h.row_ptr.assign(row_ptr, row_ptr + n + 1);
        h.col.assign(col, col + m);
        h.group.resize((size_t)n);
        for (int32_t v = 0; v < n; ++v) h.group[v] = group_of ? group_of[v] : v;
        __int128 tw = host_longest(h, [&](int32_t v) {
            int64_t x = 0;
            for (int l = 0; l < L; ++l) x = std::max(x, lat[(size_t)v * L + l]);
            return (__int128)x;
        });
        __int128 tb = host_longest(h, [&](int32_t v) {
            int64_t x = lat[(size_t)v * L];
            for (int l = 1; l < L; ++l) x = std::min(x, lat[(size_t)v * L + l]);
            return (__int128)x;
        });
        if (tw >= ((__int128)1 << 62)) return EMO_E_OVERFLOW;
        h.T_worst = (int64_t)tw;
        h.T_best = (int64_t)tb;
        int lanes = (int)((flags >> 8) & 0xFF);
        int look = (int)((flags >> 16) & 0xFF);
        std::string err;
        // backward first: the forward entries name the row of the backward program that will read
        // the node's earliest start
        // (each direction picks its own number of lanes from its ops and depth unless one is forced)
        // The distance between the group barriers: the longest of 32, 16, 8 steps that costs few slots
        // (a barrier makes every warp of a group wait for the slowest; slots take shared memory from
        // the stages).  Measured on the 250 000-node workload: forward 18 / 26 / 37 slots and
        // 11.2 / 10.5 / 10.0 ms with 8 / 16 / 32, backward 82 slots and 20.4 ms with 8, 24.5 ms with 16.
        auto compile_dir = [&](bool backward, const std::vector<uint32_t> *row_in_other, Program &out) {
            int rc = EMO_E_UNSUPPORTED;
            for (int sync = 32; sync >= 8; sync /= 2) {
                Program cand;
                rc = compile_program(h, lat, energy, backward, lanes, look, sync, row_in_other, cand, err);
                if (rc != EMO_OK && rc != EMO_E_UNSUPPORTED) return rc;
                if (rc == EMO_OK && (cand.slots <= kManySlots || sync == 8)) {
                    out = std::move(cand);
                    return EMO_OK;
                }
            }
            return rc;
        };
        // (what ends the block early, an exception among it, waits for them: they come behind what their threads use)
        struct Helper {
            std::thread t;
            void wait() { if (t.joinable()) t.join(); }
            ~Helper() { wait(); }
        };
        auto start = [](Helper &helper, auto work) {
            try {
                helper.t = std::thread(work);
            } catch (const std::exception &) {      // no more threads: here, one after the other
                work();
            }
        };
        constexpr uint32_t kTestOom = EMO_F_HOST_ONLY | EMO_F_GENERIC | EMO_F_TEST_LONG_OOM;
        const bool test_oom = flags == kTestOom;
        GraphBounds bounds;
        if (!(flags & EMO_F_GENERIC) || test_oom) graph_bounds(h, lat, energy, bounds);
        // the contracted graph, beside everything else (not where the caller shapes the programs)
        int device = 0;
        Helper joined_thread;
        if (!inner && n >= 2000 && (test_oom || (flags == 0 && cudaGetDevice(&device) == cudaSuccess)))
            start(joined_thread, [&, device]() {
                try {
                    if (test_oom) std::this_thread::sleep_for(std::chrono::milliseconds(100));
                    Contracted c;
                    contract_forward(h, lat, energy, bounds, false, c);
                    // where it leaves three nodes of five (measured, forward, us: 75 000 nodes to 11 088 x 10 001 policies 520 / 1 271; with
                    // four of five left a call gains 7 % and a load pays the second set of programs)
                    if ((int64_t)c.n * 5 > (int64_t)n * 3 || cudaSetDevice(device) != cudaSuccess) return;
                    if (load_graph(c.n, c.row_ptr.data(), c.col.data(), nullptr, 0, L, c.lat.data(), c.energy.data(), c.group.data(), flags, true, &joined.g) != EMO_OK)
                        joined.g = nullptr;
                } catch (const std::exception &) {      // no memory for it: the graph itself serves
                }
            });
        int rc = test_oom ? EMO_E_OOM : (flags & EMO_F_GENERIC) ? EMO_E_UNSUPPORTED : (inner ? EMO_OK : compile_dir(true, nullptr, g->bwd));
        if (rc == EMO_OK && !inner) rc = compile_dir(false, &g->bwd.pos_of_node, g->fwd);
        if (rc == EMO_E_UNSUPPORTED) {
            // more live exchanged values than the on-chip schedules can hold: the generic kernels take the graph
            g->generic = true;
            g->fwd = Program();
            g->bwd = Program();
            g->host_lat.assign(lat, lat + (size_t)n * L);
            g->host_energy.assign(energy, energy + (size_t)n * L);
            rc = EMO_OK;
        }
        if (rc != EMO_OK) return rc;
        if (!g->generic) {
            // stage length: the longest of 32, 16, 8 steps whose entries the producers can index
            // (32 * kFlowRowRegs per stage); one barrier per stage unless the caller says otherwise (measured on the
            // 250 000-node workload with 16 384 policies: 8 / 16 / 32 steps between barriers gave 24.8 / 22.3 / 21.3 ms for
            // both passes)
            int fk = (int)((flags >> 24) & 0x3F), fs = (int)((flags >> 4) & 0xF) * 8;
            int flanes = g->fwd.lanes > 0 ? std::max(g->fwd.lanes, g->bwd.lanes) : 1;
            if (inner) flanes = pick_lanes(n, hop_depth(h));
            if (fk == 0) fk = flanes * 32 <= 32 * kFlowRowRegs ? 32 : (flanes * 16 <= 32 * kFlowRowRegs ? 16 : 8);
            if (fs == 0) fs = fk;
            if (fs > fk) fs = fk;
            // the spine program: short stages (its sums per stage live in shared memory), 16 steps unless the caller
            // says otherwise; compiled on a thread of its own beside the lane-stream program (they share nothing but
            // their inputs)
            const bool want_spine = !(flags & EMO_F_INTERVALS);
            // the slice program, for calls with few policies: another thread (not where the caller shapes the spine program)
            const bool want_slices = want_spine && !(flags & (EMO_F_HOST_ONLY | 0xC0000000u));
            int rc_s = EMO_OK, rc_l = EMO_E_UNSUPPORTED;
            std::string err_s, err_l;
            Helper spine_thread, long_thread, slice_thread, walk_thread;
            const bool no_long = (flags & EMO_F_TEST_LONG_OOM) != 0 && (flags & EMO_F_HOST_ONLY) != 0;
            auto compile_spine = [&](int k, Flow &out, DevSpine &d, SpineImage &im, int &rc_k, std::string &err_k) {
                try {
                    if (no_long && &out == &g->lflow) throw std::bad_alloc();
                    rc_k = compile_flow(h, lat, energy, bounds, lanes, look, k, k, out, err_k, true);
                    if (rc_k == EMO_OK) rc_k = lay_out_spine(out, d, im);
                } catch (const std::bad_alloc &) {
                    rc_k = EMO_E_OOM;
                } catch (const std::exception &) {
                    rc_k = EMO_E_UNSUPPORTED;
                }
            };
            if ((flags & EMO_F_INTERVALS) && !(flags & EMO_F_HOST_ONLY))
                start(walk_thread, [&]() {
                    try {
                        compile_walk(h, lat, energy, bounds, g->walk);
                    } catch (const std::exception &) {      // no memory for it: the others serve
                        g->walk = Walk();
                    }
                });
            if (want_slices)
                start(slice_thread, [&]() {
                    try {
                        compile_slices(h, lat, energy, bounds, slices);
                    } catch (const std::exception &) {      // no memory for it: the others serve
                        slices = Slices();
                    }
                });
            if (want_spine) {
                const int code = (int)((flags >> 30) & 3u);
                // Measured (forward + backward, ms): 18 lanes, 128 039 nodes x 8 192 policies 6.2 with 4 positions, 6.6 with 5
                // and 8.9 with 8 (a stage of 8 leaves room for one buffer less); 4 lanes, 250 000 x 16 384 15.0 with
                // 16, 17.2 with 12; 1 013 x 65 536 0.36 with 16, 0.48 with 20 and 0.43 with 8.
                int sk = code == 1 ? 8 : (code == 3 ? 32 : (code == 2 || flanes <= 8 ? 16 : 4));
                while (sk > 8 && flanes * sk > 32 * kFlowRowRegs) sk /= 2;
                start(spine_thread, [&, sk]() { compile_spine(sk, g->sflow, g->dspine, g->simage, rc_s, err_s); });
                // the long stages: as many positions as make about a hundred entries (ms, both passes: 25 000 nodes, 5 lanes x 2 000
                // policies: 20 positions 0.78, 16 0.83; 10 000, 3 lanes x 4 096: 32 0.60, 24 0.66); more than eight lanes about 126, the
                // seven positions that were best on the one wide graph measured (51 000, 18 lanes x 1 000: 7 1.82, 6 1.90, 5 1.96)
                const int lk = std::min(32, (flanes > 8 ? 126 : 100) / flanes);
                if (code == 0 && lk > sk)
                    start(long_thread, [&, lk]() { compile_spine(lk, g->lflow, g->dlong, g->limage, rc_l, err_l); });
            }
            try {
                if (!inner) rc = compile_flow(h, lat, energy, bounds, lanes, look, fk, fs, g->flow, err);
            } catch (const std::bad_alloc &) {
                rc = EMO_E_OOM;
            }
            spine_thread.wait();
            long_thread.wait();
            slice_thread.wait();
            walk_thread.wait();
            if (rc == EMO_E_UNSUPPORTED) {      // the 64-bit programs exist: they serve
                g->flow = Flow();
                rc = EMO_OK;
            }
            if (rc == EMO_OK && rc_s != EMO_OK && rc_s != EMO_E_UNSUPPORTED) rc = rc_s;
            if (rc != EMO_OK) return rc;
            if (!want_spine || rc_s != EMO_OK || !(g->flow.ok32 || inner) || !g->sflow.spine.ok) g->sflow = Flow();
            else {
                // only the spine's parts are kept
                g->sflow.f = FlowDir();
                g->sflow.b = FlowDir();
            }
            // (a tail is folded only over a distance of two stages: where long stages leave fewer folds the program has more
            // operations, and the short one is faster: 25 000 nodes with 21 positions 59 000 operations, 1.7 ms, with 20 15 000, 0.78 ms)
            auto operations = [](const Spine &s2) {
                int64_t c = 0;
                for (uint32_t k : s2.f.n_ops) c += k;
                for (uint32_t k : s2.b.n_ops) c += k;
                return c;
            };
            // (nor is it there when memory did not suffice for it: every call has the short one)
            if (rc_l != EMO_OK || !g->sflow.spine.ok || !g->lflow.spine.ok || operations(g->lflow.spine) > operations(g->sflow.spine) * 5 / 4) g->lflow = Flow();
            g->lflow.f = FlowDir();
            g->lflow.b = FlowDir();
        }
        h.depth = hop_depth(h);
        joined_thread.wait();
        if (!g->generic) std::swap(g->joined, joined.g);
    } catch (const std::bad_alloc &) {
        return EMO_E_OOM;
    }
    if (g->host_only) {
        g->dspine.ready = g->sflow.spine.ok && !g->simage.host.empty();
        g->dlong.ready = g->lflow.spine.ok && !g->limage.host.empty();
    } else {
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess) { (void)cudaGetLastError(); return EMO_E_CUDA; }
        // (two attributes; all of a device's properties take 3 to 10 ms, more than everything else for a small graph)
        int sms = 0, shared = 0;
        if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&shared, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess) {
            (void)cudaGetLastError();
            return EMO_E_CUDA;
        }
        g->device = dev;
        g->sm_count = sms;
        g->smem_optin = (size_t)shared;
        int rc = EMO_OK;
        try {
        if (g->generic) {
            // successor CSR from the predecessor CSR, then everything the generic kernels read
            const HostGraph &hh = g->h;
            std::vector<int64_t> sp((size_t)hh.n + 1, 0);
            std::vector<int32_t> sc((size_t)std::max<int64_t>(hh.m, 1));
            for (int64_t e = 0; e < hh.m; ++e) sp[(size_t)hh.col[e] + 1]++;
            for (int32_t v = 0; v < hh.n; ++v) sp[(size_t)v + 1] += sp[(size_t)v];
            std::vector<int64_t> fill(sp.begin(), sp.end() - 1);
            for (int32_t v = 0; v < hh.n; ++v)
                for (int64_t e = hh.row_ptr[v]; e < hh.row_ptr[v + 1]; ++e) sc[(size_t)fill[(size_t)hh.col[e]]++] = v;
            rc = upload(&g->gen_row_ptr, hh.row_ptr.data(), hh.row_ptr.size() * 8);
            if (rc == EMO_OK) rc = upload(&g->gen_col, hh.col.data(), hh.col.size() * 4);
            if (rc == EMO_OK) rc = upload(&g->gen_srow_ptr, sp.data(), sp.size() * 8);
            if (rc == EMO_OK) rc = upload(&g->gen_scol, sc.data(), (size_t)hh.m * 4);
            if (rc == EMO_OK) rc = upload(&g->gen_group, hh.group.data(), hh.group.size() * 4);
            if (rc == EMO_OK) rc = upload(&g->gen_lat, g->host_lat.data(), g->host_lat.size() * 8);
            if (rc == EMO_OK) rc = upload(&g->gen_energy, g->host_energy.data(), g->host_energy.size() * 8);
            g->host_lat = std::vector<int64_t>();
            g->host_energy = std::vector<double>();
        } else {
        if (!inner) rc = upload_program(g->fwd, g->dfwd);
        if (rc == EMO_OK && !inner) rc = upload_program(g->bwd, g->dbwd);
        if (rc == EMO_OK && !inner && g->fwd.lanes <= 32 - kProducerWarps && g->bwd.lanes <= 32 - kProducerWarps) {
            rc = upload_program_lane(g->fwd, g->lfwd);
            if (rc == EMO_OK) rc = upload_program_lane(g->bwd, g->lbwd);
        }
        if (rc == EMO_OK && !inner) rc = upload_flow(g->flow, g->dflow, (flags & EMO_F_INTERVALS) != 0);
        // One barrier per stage needs more exchange slots than one every 16 steps (on the 250 000-node graph 20.9 KB
        // against 13.8 KB per policy group, at 0.3 scale 29.8 KB against 17.9 KB).  Where four groups then no longer fit a
        // block, the grid doubles and the gain turns into a loss (11.7 ms against 6.8 ms at 0.3 scale): take the shorter
        // distance unless the caller chose one.
        if (rc == EMO_OK && g->flow.ok32 && g->dflow.ready && !(flags & 0xF0u) && g->flow.sync > 16) {
            FlowPlan probe;
            const int gmax = std::min((32 - 2) / std::max(g->flow.lanes, 1), 15);
            const bool fits = flow_plan(g, (int64_t)4 * 32 * g->sm_count - 1, true, true, probe) && probe.groups >= std::min(4, gmax);
            if (!fits) {
                const int fk = g->flow.K, look = (int)((flags >> 16) & 0xFF);
                int lanes = (int)((flags >> 8) & 0xFF);
                std::string err;
                free_flow(g->dflow);
                GraphBounds bounds;
                graph_bounds(g->h, lat, energy, bounds);
                rc = compile_flow(g->h, lat, energy, bounds, lanes, look, fk, 16, g->flow, err);
                if (rc == EMO_E_UNSUPPORTED) {
                    g->flow = Flow();
                    rc = EMO_OK;
                }
                if (rc == EMO_OK) rc = upload_flow(g->flow, g->dflow, (flags & EMO_F_INTERVALS) != 0);
            }
        }
        if (rc == EMO_OK && g->sflow.spine.ok) rc = upload_spine(g->simage, g->dspine);
        if (rc == EMO_OK && g->lflow.spine.ok) {
            const int rc_l = (flags & EMO_F_TEST_LONG_OOM) ? EMO_E_OOM : upload_spine(g->limage, g->dlong);
            if (rc_l == EMO_OK) keep_sizes(g->lflow);
            else if (rc_l == EMO_E_OOM) g->lflow = Flow();      // the short program serves every call
            else rc = rc_l;
        }
        g->simage = g->limage = SpineImage();
        if (rc == EMO_OK && g->walk.ok) {
            const int rc_w = upload(&g->dwalk, g->walk.blob.data(), g->walk.blob.size());
            if (rc_w != EMO_OK && rc_w != EMO_E_OOM) rc = rc_w;
            g->walk.ok = rc_w == EMO_OK;
            g->walk.blob = std::vector<unsigned char>();
        }
        if (rc == EMO_OK && slices.ok) {
            // (nodes with very many operands: a slice's steps, or its matrices, that no block's shared memory holds)
            size_slices(slices, g->dslice);
            SlicePlan probe;
            const bool fits = slice_plan(g, 1, false, false, 0, probe) || slice_plan(g, 1, false, false, 1, probe);
            if (!fits) g->dslice = DevSlice();
            const int rc_c = fits ? upload_slices(slices, g->dslice) : EMO_OK;
            if (rc_c != EMO_OK && rc_c != EMO_E_OOM) rc = rc_c;      // (no memory for it: the others serve)
        }
        }
        } catch (const std::bad_alloc &) {
            rc = EMO_E_OOM;
        }
        if (rc != EMO_OK) return rc;
        if (!inner) g->one_bytes = pass_ws_bytes(g, 1, 1, 0, 1);
    }
    owned.g = nullptr;
    *out = g;
    return EMO_OK;
}

int emo_graph_load(int32_t n, const int64_t *row_ptr, const int32_t *col, const int32_t *level_ptr,
                   int32_t n_levels, int32_t L, const int64_t *lat, const double *energy,
                   const int32_t *group_of, uint32_t flags, emo_graph **out)
{
    return load_graph(n, row_ptr, col, level_ptr, n_levels, L, lat, energy, group_of, flags, false, out);
}

int emo_graph_free(emo_graph *g)
{
    if (!g) return EMO_OK;
    emo_graph_free(g->joined);
    if (!g->host_only) {
        free_program(g->dfwd);
        free_program(g->dbwd);
        free_program_lane(g->lfwd);
        free_program_lane(g->lbwd);
        free_flow(g->dflow);
        free_spine(g->dspine);
        free_spine(g->dlong);
        if (g->dslice.mem) cudaFree(g->dslice.mem);
        if (g->dwalk) cudaFree(g->dwalk);
        void *gen[] = {g->gen_row_ptr, g->gen_col, g->gen_srow_ptr, g->gen_scol, g->gen_group, g->gen_lat, g->gen_energy};
        for (void *q : gen)
            if (q) cudaFree(q);
    }
    delete g;
    return EMO_OK;
}

int emo_graph_info(const emo_graph *g, emo_info *info)
{
    if (!g || !info) return EMO_E_INVALID_ARG;
    info->n = g->h.n;
    info->m = g->h.m;
    info->L = g->h.L;
    info->rows = g->h.rows;
    info->depth = g->h.depth;
    info->max_span = g->h.max_span;
    info->T_worst = g->h.T_worst;
    info->T_best = g->h.T_best;
    info->lanes = g->fwd.lanes;
    info->lanes_bwd = g->bwd.lanes;
    info->sync_fwd = g->fwd.sync;
    info->sync_bwd = g->bwd.sync;
    info->steps_fwd = g->fwd.steps;
    info->slots_fwd = g->fwd.slots;
    info->aux_fwd = g->fwd.aux;
    info->steps_bwd = g->bwd.steps;
    info->slots_bwd = g->bwd.slots;
    info->aux_bwd = g->bwd.aux;
    return EMO_OK;
}

int emo_graph_flow(const emo_graph *g, emo_flow_view *v)
{
    if (!g || !v) return EMO_E_INVALID_ARG;
    const Flow &f = g->flow;
    std::memset(v, 0, sizeof *v);
    v->ok32 = f.ok32 ? 1 : 0;
    v->lanes = f.lanes;
    v->K = f.K;
    v->sync = f.sync;
    v->stages = f.stages;
    v->steps = f.steps;
    v->Lp = f.Lp;
    v->slots_tag_fwd = f.f.slots_tag;
    v->slots_set_fwd = f.f.slots_set;
    v->pool_stride_fwd = f.f.pool_stride;
    v->slots_tag_bwd = f.b.slots_tag;
    v->slots_set_bwd = f.b.slots_set;
    v->pool_stride_bwd = f.b.pool_stride;
    v->pushes = f.pushes;
    v->pruned_fwd = f.f.pruned;
    v->pruned_bwd = f.b.pruned;
    v->hdr = f.hdr.data();
    v->rows = f.rows.data();
    v->node = f.node.data();
    v->step = f.step.data();
    v->tab_fwd = f.tabF.data();
    v->tab_bwd = f.tabB.data();
    v->rec_fwd = f.f.rec.data();
    v->pool_fwd = f.f.pool.data();
    v->rec_bwd = f.b.rec.data();
    v->pool_bwd = f.b.pool.data();
    v->seg_fwd = f.f.seg.data();
    v->seg_bwd = f.b.seg.data();
    v->lbes = f.lbes.data();
    v->push_base = f.push_base.data();
    return EMO_OK;
}

int emo_graph_spine(const emo_graph *g, int64_t out[12])
{
    if (!g || !out) return EMO_E_INVALID_ARG;
    for (int i = 0; i < 12; ++i) out[i] = 0;
    const Flow &f = g->sflow;
    if (!f.ok32 || !f.spine.ok) return EMO_OK;
    int64_t nf = 0, nb = 0;
    for (uint32_t c : f.spine.f.n_ops) nf += c;
    for (uint32_t c : f.spine.b.n_ops) nb += c;
    const int64_t v[12] = {1, f.lanes, f.K, f.stages, f.spine.segments, nf, nb, f.spine.f.slots, f.spine.b.slots,
                           f.spine.max_segs, f.spine.acc_words, f.spine.pushes};
    for (int i = 0; i < 12; ++i) out[i] = v[i];
    return EMO_OK;
}

int emo_graph_spine_plan(const emo_graph *g, int64_t B, int need_slack, int want_base, int32_t sm_count, int64_t smem_bytes, int64_t out[12])
{
    if (!g || !out || B < 0 || sm_count < 1 || smem_bytes < 0) return EMO_E_INVALID_ARG;
    for (int i = 0; i < 12; ++i) out[i] = 0;
    SpinePlan pl;
    if (!spine_plan_on(g, SpineChip{sm_count, (size_t)smem_bytes}, B, want_base != 0, need_slack != 0, need_slack > 1, pl)) return EMO_OK;
    const Flow &f = pl.is_long ? g->lflow : g->sflow;
    const int64_t v[12] = {1, pl.is_long ? 1 : 0, f.lanes, f.K, f.stages, f.spine.bundle, pl.k->nb, pl.k->max_threads, pl.groups, pl.vw, pl.vs,
                           std::max(pl.threads_f, pl.threads_b)};
    for (int i = 0; i < 12; ++i) out[i] = v[i];
    return EMO_OK;
}

int emo_graph_spine_view(const emo_graph *g, emo_spine_view *v)
{
    if (!g || !v) return EMO_E_INVALID_ARG;
    std::memset(v, 0, sizeof *v);
    const Flow &f = g->sflow;
    const Spine &sp = f.spine;
    if (!f.ok32 || !sp.ok) return EMO_OK;
    v->ok = 1;
    v->lanes = f.lanes;
    v->K = f.K;
    v->stages = f.stages;
    v->Lp = f.Lp;
    v->max_ops_fwd = sp.f.max_ops;
    v->max_ops_bwd = sp.b.max_ops;
    v->max_pool = sp.max_pool;
    v->acc_words = sp.acc_words;
    v->slots_fwd = sp.f.slots;
    v->slots_bwd = sp.b.slots;
    v->pushes = sp.pushes;
    v->n_ops_fwd = sp.f.n_ops.data();
    v->ops_fwd = sp.f.ops.data();
    v->n_ops_bwd = sp.b.n_ops.data();
    v->ops_bwd = sp.b.ops.data();
    v->mem = sp.mem.data();
    v->pos = sp.posw.data();
    v->rows = f.rows.data();
    v->tab_fwd = f.tabF.data();
    v->tab_bwd = f.tabB.data();
    v->pool = sp.pool.data();
    v->push_base = sp.push_base.data();
    return EMO_OK;
}

int emo_graph_spine_layout(const emo_graph *g, int long_program, emo_spine_layout *v)
{
    if (!g || !v || (long_program != 0 && long_program != 1)) return EMO_E_INVALID_ARG;
    std::memset(v, 0, sizeof *v);
    const Flow &f = long_program ? g->lflow : g->sflow;
    const DevSpine &d = long_program ? g->dlong : g->dspine;
    const SpineImage &im = long_program ? g->limage : g->simage;
    if (!f.ok32 || !f.spine.ok || im.host.empty()) return EMO_OK;
    v->ok = 1;
    v->lanes = f.lanes;
    v->stages = f.stages;
    v->Lp = f.Lp;
    v->bundle = f.spine.bundle;
    v->nlook = d.nlook;
    v->chunks = d.chunks;
    v->most_chunks = kSpChunks;
    v->max_segs = f.spine.max_segs;
    v->unread_slot = (int32_t)f.spine.unread_slot;
    v->slots_fwd = f.spine.f.slots;
    v->slots_bwd = f.spine.b.slots;
    v->pushes = f.spine.pushes;
    const DevSpineDir *dir[2] = {&d.f, &d.b};
    for (int k = 0; k < 2; ++k) {
        v->w_bytes[k] = (int32_t)dir[k]->w_bytes;
        v->s_bytes[k] = (int32_t)dir[k]->s_bytes;
        v->off_pos[k] = (int32_t)dir[k]->off_pos;
        v->off_tab[k] = (int32_t)dir[k]->off_tab;
        v->off_ops[k] = (int32_t)dir[k]->off_ops;
        v->off_rec[k] = (int32_t)dir[k]->off_rec;
        v->words[k] = dir[k]->words;
        v->zero[k] = dir[k]->zero;
        v->w[k] = im.host.data() + (k ? im.at_bW : im.at_fW);
        v->s[k] = im.host.data() + (k ? im.at_bS : im.at_fS);
        v->rows[k] = (const uint32_t *)(im.host.data() + (k ? im.at_rowsB : im.at_rowsF));
    }
    v->off_mem = (int32_t)d.b.off_mem;
    v->off_first = (int32_t)d.b.off_first;
    v->push_base = (const uint32_t *)(im.host.data() + im.at_pb);
    return EMO_OK;
}

int emo_graph_program(const emo_graph *g, int dir, int32_t *lanes, int32_t *steps, int32_t *slots,
                      int32_t *Lp, const uint32_t **entries, const uint32_t **rows, const uint32_t **lat)
{
    if (!g || (dir != 0 && dir != 1)) return EMO_E_INVALID_ARG;
    const Program &p = dir ? g->bwd : g->fwd;
    if (lanes) *lanes = p.lanes;
    if (steps) *steps = p.steps;
    if (slots) *slots = p.slots;
    if (Lp) *Lp = p.Lp;
    if (entries) *entries = p.entries.data();
    if (rows) *rows = p.rows.data();
    if (lat) *lat = p.lat.data();
    return EMO_OK;
}

}  // extern "C"

namespace {

// Spill area behind the head of the workspace: large enough for either layout.
size_t spill_need(const emo_graph *g, int64_t B)
{
    size_t plain = (size_t)g->h.n * round_up((size_t)B, 16) * sizeof(int64_t);
    size_t tiled = 0;
    if (!g->host_only && B > 0) {
        LaunchShape s;
        StagedParams sp;
        // either staged kernel may run (the call's flags decide): room for the wider tiling
        for (int which = 0; which < 2; ++which) {
            const bool ok = which ? staged_shape(g, g->bwd, g->dbwd.rec_bytes, true, B, s, sp) : lane_shape(g, g->bwd, true, B, s, sp);
            if (!ok) continue;
            const size_t tiles = ((size_t)B + sp.ptile - 1) / sp.ptile;
            tiled = std::max(tiled, tiles * spill_rows_of(g, which == 0) * sp.ptile * sizeof(int64_t));
        }
    }
    return round_up(std::max(plain, tiled), 256);
}

}  // namespace

extern "C" {

// The generic kernels: completion times (and, for the backward pass, tails) of every node in the workspace.
static size_t generic_need(const emo_graph *g, int64_t B, bool need_bwd)
{
    const size_t ldw = round_up((size_t)B + 1, 16);
    return (size_t)std::max(g->h.n, 1) * ldw * 8 * (need_bwd ? 2 : 1);
}

static int launch_generic(const emo_graph *g, int64_t B, const uint8_t *lvl, int64_t ldb, bool need_bwd, int64_t *ES, int64_t *LS,
                          int64_t *slack, int64_t ldo, int64_t *makespan, double *energy, int64_t *slack_sum, int32_t *n_critical,
                          int64_t *T0, double *E0, void *ws, size_t ws_bytes, cudaStream_t st)
{
    const size_t head = kSmallWs + lvl_area(g);
    if (!ws || ws_bytes < head + generic_need(g, B, need_bwd)) return EMO_E_OOM;
    GenericParams p;
    p.n = g->h.n;
    p.L = g->h.L;
    p.row_ptr = g->gen_row_ptr;
    p.col = g->gen_col;
    p.srow_ptr = g->gen_srow_ptr;
    p.scol = g->gen_scol;
    p.group = g->gen_group;
    p.lat = g->gen_lat;
    p.energy = g->gen_energy;
    p.B = B;
    p.want_base = (T0 || E0) ? 1 : 0;
    p.lvl = lvl;
    p.ldb = ldb;
    p.ldw = (int64_t)round_up((size_t)B + 1, 16);
    p.C = (int64_t *)((char *)ws + head);
    p.Q = p.C + (size_t)std::max(g->h.n, 1) * p.ldw;
    p.ES = ES;
    p.LS = LS;
    p.slack = slack;
    p.ldo = ldo;
    p.makespan = makespan;
    p.energy_out = energy;
    p.slack_sum = slack_sum;
    p.n_critical = n_critical;
    p.base_T = T0;
    p.base_E = E0;
    const int64_t cols = B + p.want_base;
    if (cols == 0) return EMO_OK;
    cudaEvent_t ev0 = g_pass_events[0], ev1 = g_pass_events[1], ev2 = g_pass_events[2], ev3 = g_pass_events[3];
    if (ev0) EMO_CUDA(cudaEventRecord(ev0, st));
    emo_generic_fwd<<<(unsigned)((cols + 127) / 128), 128, 0, st>>>(p);
    EMO_CUDA(cudaGetLastError());
    if (ev1) EMO_CUDA(cudaEventRecord(ev1, st));
    if (need_bwd && B > 0) {
        if (ev2) EMO_CUDA(cudaEventRecord(ev2, st));
        emo_generic_bwd<<<(unsigned)((B + 127) / 128), 128, 0, st>>>(p);
        EMO_CUDA(cudaGetLastError());
        if (ev3) EMO_CUDA(cudaEventRecord(ev3, st));
    }
    return EMO_OK;
}

// Workspace of the pass kernels (a call with less than that is refused; the slice kernels' share is only for their use).
static size_t pass_ws_bytes(const emo_graph *g, int64_t B, int need_slack, uint32_t flags, int aligned)
{
    size_t bytes = kSmallWs + lvl_area(g);
    if (g->generic) {
        bytes += generic_need(g, B, need_slack != 0);
        return bytes;
    }
    if (need_slack) {
        // what the call with these flags will run: the 32-bit kernels keep a restore list between the
        // passes, the 64-bit kernels the earliest starts of every node
        size_t need = 0;
        FlowPlan fp;
        const uint8_t *fake = aligned ? (const uint8_t *)16 : (const uint8_t *)1;
        if (!g->host_only && B > 0 && flow_allowed(g, B, fake, aligned ? 16 : 1, 0, flags) && flow_plan(g, B, true, true, fp))
            need = fp.restore_bytes;
        else
            need = spill_need(g, B);
        SpinePlan sp;
        if (!g->host_only && B > 0 && spine_allowed(g, B, fake, aligned ? 16 : 1, 0, flags) && spine_plan(g, B, true, true, false, sp))
        {
            // (rows of the larger of the two programs and, where tiles are larger than two groups, up to seven groups more: a smaller
            // batch, or a call with other outputs, may take the other program or a larger tile)
            const size_t cover = (size_t)sp.grid_f * (size_t)sp.groups, groups = cover + (cover > 2 * (size_t)g->sm_count ? 7 : 0);
            need = std::max(need, groups * 128 * (size_t)std::max(sp.pf.restore_rows, g->lflow.spine.pushes + g->lflow.lanes) + 256);
        }
        bytes += need;
    }
    return bytes;
}

int emo_workspace_bytes_for(const emo_graph *g, int64_t B, int need_slack, uint32_t flags, int aligned, size_t *out)
{
    if (!g || !out || B < 0) return EMO_E_INVALID_ARG;
    size_t bytes = pass_ws_bytes(g, B, need_slack, flags, aligned);
    const emo_graph *const joined = need_slack ? nullptr : joined_for(g, flags);
    bytes = std::max(bytes, kSmallWs + lvl_area(g) + slice_call_ws(joined ? joined : g, B, need_slack != 0, flags));
    if (need_slack == 2) bytes += 4 * round_up((size_t)B * 8, 256) + 256;
    *out = bytes;
    return EMO_OK;
}

int emo_workspace_bytes(const emo_graph *g, int64_t B, int need_slack, size_t *out)
{
    return emo_workspace_bytes_for(g, B, need_slack, 0, 1, out);
}

int emo_eval_policies(const emo_graph *g, int64_t B, const uint8_t *lvl, int64_t ldb, int64_t *makespan,
                      double *energy, int64_t *T0, double *E0, void *ws, size_t ws_bytes, int32_t *status,
                      uint32_t flags, void *stream)
{
    if (!g || B < 0) return EMO_E_INVALID_ARG;
    if (g->host_only) return EMO_E_CUDA;
    if (B == 0 && !T0 && !E0) return EMO_OK;
    if (B > 0 && (!lvl || !makespan || !energy || ldb < B)) return EMO_E_INVALID_ARG;
    cudaStream_t st = (cudaStream_t)stream;
    if ((flags & EMO_F_VALIDATE) && B > 0) {
        int rc = launch_validate(g, B, lvl, ldb, status, st);
        if (rc) return rc;
    }
    if (B == 0) { lvl = nullptr; ldb = 0; }
    if (g->generic)
        return launch_generic(g, B, lvl, ldb, false, nullptr, nullptr, nullptr, 0, makespan, energy, nullptr, nullptr, T0, E0, ws,
                              ws_bytes, st);
    const size_t head = kSmallWs + lvl_area(g);
    for (const emo_graph *e : {joined_for(g, flags), g}) {
        if (!e) continue;
        int rc = EMO_OK;
        if (slice_call(e, B, false, flags, {lvl, ldb, nullptr, nullptr, nullptr, 0, makespan, energy, nullptr, nullptr, T0, E0}, ws, ws_bytes, head, st, rc)) return rc;
        SpinePlan fp;
        if (spine_allowed(e, B, lvl, ldb, 0, flags) && spine_plan(e, B, T0 || E0, false, false, fp))
            return launch_spine_fwd(e, fp, B, lvl, ldb, nullptr, makespan, energy, T0, E0, status, flags, st);
    }
    if (flow_allowed(g, B, lvl, ldb, 0, flags)) {
        FlowPlan fp;
        if (flow_plan(g, B, T0 || E0, false, fp))
            return launch_flow_fwd(g, fp, B, lvl, ldb, nullptr, makespan, energy, T0, E0, status, flags, st);
    }
    PassPlan pl;
    int rc = make_plan(g, B, T0 || E0, false, lvl, ldb, 0, 0, flags, pl);
    if (rc) return rc;
    return launch_pass(g, pl, false, B, lvl, ldb, nullptr, 0, nullptr, nullptr, nullptr, 0, makespan, energy, nullptr,
                       nullptr, T0, E0, status, st);
}

int emo_workspace_bytes_intervals(const emo_graph *g, int64_t B, int32_t I, int with_idle, size_t *out)
{
    if (!g || !out || B < 0 || I < 1) return EMO_E_INVALID_ARG;
    size_t bytes = round_up((size_t)I * 8, 256);
    if (with_idle) bytes += (size_t)std::max(g->h.rows, 1) * (size_t)I * round_up((size_t)B, 16) * 8;
    *out = bytes;
    return EMO_OK;
}

// The shape of a call that the walk kernel takes: a uniform grid, the columns of F in shared memory.
static bool walk_plan(const emo_graph *g, int64_t B, int rows, int32_t I, int64_t delta, WalkParams &p, int &grid, size_t &smem)
{
    const Walk &w = g->walk;
    if (!w.ok || delta <= 0 || delta >= kWalkMaxDur) return false;
    p = WalkParams();
    p.blob = g->dwalk;
    p.chunks = w.chunks;
    p.Lp = w.Lp;
    p.L = g->h.L;
    p.chunk_bytes = w.chunk_bytes;
    p.off_dur = w.off_dur;
    p.off_en = w.off_en;
    p.rows = rows;
    p.I = I;
    p.B = B;
    p.delta = (int)delta;
    p.inv = 1.0f / (float)delta;
    p.energy0 = w.energy0;
    // fewer policies per warp as long as every warp has a scheduler of its own (fewer of them leave an interval inside an item); then
    // as many warps per block as bring all in at once
    int64_t pl = 4;
    while (pl < 32 && (B + pl - 1) / pl > (int64_t)g->sm_count * 4) pl *= 2;
    const int64_t warps = (B + pl - 1) / pl;
    int groups = (int)std::min<int64_t>(kWalkMaxGroups, (warps + g->sm_count - 1) / g->sm_count);
    for (; groups >= 1; --groups) {
        p.groups = groups;
        p.pl = (int)pl;
        p.P = groups * (int)pl;
        p.off_F = 2 * kWalkMaxBuffers * 8 + 16;
        const size_t f_bytes = (size_t)rows * (size_t)I * (size_t)p.P, off_slots = round_up(p.off_F + f_bytes, 128);
        const size_t off_buf = round_up(off_slots + (size_t)w.slots * groups * 256, 128);
        for (p.buffers = kWalkMaxBuffers; p.buffers >= 2; --p.buffers) {
            smem = off_buf + (size_t)p.buffers * w.chunk_bytes;
            if (smem > g->smem_optin) continue;
            p.off_slots = (unsigned)off_slots;
            p.off_buf = (unsigned)off_buf;
            grid = (int)((B + p.P - 1) / p.P);
            return true;
        }
    }
    return false;
}

// Whether the walk kernel is the faster one.  Measured (us, it / the lane-stream kernel, 26 intervals): up to three lanes, 500 nodes x 4 096
// policies 67 / 173, 10 000 x 16 384 1 899 / 2 408; more lanes in one wave of blocks against two or more, 18 lanes, 38 000 nodes x
// 16 384 2 212 / 6 161, 5 lanes, 25 000 x 40 000 2 184 / 2 834; not in one against one, 75 000 x 16 384 (80 intervals) 5 462 / 3 795, 38 000 x
// 4 096 2 014 / 1 645.  Where F does not fit the lane-stream kernel's blocks it seldom suits these (8 rows, 400 intervals, 6 439 nodes x
// 16 2 065 / 1 522 by the step program).
static bool walk_pays(const emo_graph *g, int64_t B, int rows, int32_t I, int walk_grid)
{
    const int64_t sms = std::max(g->sm_count, 1), walk_waves = (walk_grid + sms - 1) / sms;
    FlowPlan fp;
    const size_t brk_b = round_up((size_t)I * 8, 16), f_per_group = (size_t)rows * (size_t)I * 32;
    if (!g->dflow.blobFI || !flow_plan(g, B, false, false, fp, true, brk_b, f_per_group)) return false;
    const int64_t flow_waves = (fp.grid_f + sms - 1) / sms;
    return g->flow.lanes <= 3 ? walk_waves <= flow_waves : walk_waves * 2 <= flow_waves;
}

// Length of the intervals of a uniform grid, else 0.
static long long interval_length(int32_t I, const int64_t *breaks)
{
    const long long delta = I > 1 ? breaks[1] : 0;
    for (int32_t i = 1; i < I && delta > 0; ++i)
        if (breaks[i] != (int64_t)i * delta) return 0;
    return delta;
}

// Which kernel evaluates a call with time intervals, and how it is launched.
enum { kIntervalSteps, kIntervalFlow, kIntervalWalk };
struct IntervalPlan {
    WalkParams walk;
    FlowPlan flow;
    int walk_grid = 0;
    size_t walk_smem = 0;
};
// walk: whether the walk kernel may take it (1), must where it can (2), or does not (0)
static int interval_kernel(const emo_graph *g, int64_t B, int32_t I, long long delta, uint32_t flags, int walk, IntervalPlan &pl)
{
    const int rows = std::max(g->h.rows, 1);
    if ((flags & EMO_F_NO_STAGING) || delta <= 0) return kIntervalSteps;
    if (walk && !(flags & EMO_F_FLOW_KERNEL) && walk_plan(g, B, rows, I, delta, pl.walk, pl.walk_grid, pl.walk_smem) &&
        (walk == 2 || walk_pays(g, B, rows, I, pl.walk_grid)))
        return kIntervalWalk;
    return g->dflow.blobFI && flow_plan(g, B, false, false, pl.flow, true, round_up((size_t)I * 8, 16), (size_t)rows * (size_t)I * 32) ? kIntervalFlow : kIntervalSteps;
}

static int eval_intervals(const emo_graph *g, int64_t B, const uint8_t *F, int64_t ldb, int32_t I, const int64_t *breaks,
                          const double *p_idle, int64_t *makespan, double *energy, double *energy_idle, void *ws,
                          size_t ws_bytes, int32_t *status, uint32_t flags, int walk, void *stream)
{
    if (!g || B < 0 || I < 1 || I > 4096 || !breaks || breaks[0] != 0) return EMO_E_INVALID_ARG;
    for (int32_t i = 1; i < I; ++i)
        if (breaks[i] <= breaks[i - 1]) return EMO_E_INVALID_ARG;
    if (g->host_only) return EMO_E_CUDA;
    if (g->generic) return EMO_E_UNSUPPORTED;      // the time-interval form needs a compiled schedule
    if (B == 0) return EMO_OK;
    if (!F || !makespan || !energy || ldb < B) return EMO_E_INVALID_ARG;
    if (energy_idle && !p_idle) return EMO_E_INVALID_ARG;
    size_t need = 0;
    emo_workspace_bytes_intervals(g, B, I, p_idle != nullptr, &need);
    if (!ws || ws_bytes < need) return EMO_E_OOM;
    cudaStream_t st = (cudaStream_t)stream;
    int64_t *d_breaks = (int64_t *)ws;
    unsigned long long *busy = p_idle ? (unsigned long long *)((char *)ws + round_up((size_t)I * 8, 256)) : nullptr;
    const int64_t ldw = (int64_t)round_up((size_t)B, 16);
    const int rows = std::max(g->h.rows, 1);
    EMO_CUDA(cudaMemcpyAsync(d_breaks, breaks, (size_t)I * 8, cudaMemcpyHostToDevice, st));
    if (busy) EMO_CUDA(cudaMemsetAsync(busy, 0, (size_t)rows * (size_t)I * (size_t)ldw * 8, st));
    const float inv_mean = (I > 1) ? (float)((double)(I - 1) / (double)breaks[I - 1]) : 0.0f;
    const long long delta = interval_length(I, breaks);
    cudaEvent_t ev0 = g_pass_events[0], ev1 = g_pass_events[1];
    if (ev0) EMO_CUDA(cudaEventRecord(ev0, st));
    IntervalPlan plan;
    const int which = interval_kernel(g, B, I, delta, flags, walk, plan);
    if (which == kIntervalWalk) {
        WalkParams &q = plan.walk;
        q.F = F;
        q.ldF = ldb;
        q.makespan = makespan;
        q.energy = energy;
        q.busy = busy;
        q.ldw = ldw;
        q.status = status;
        q.wait_cycles = g_wait_cycles;
        if (flow_optin(emo_walk, g) != EMO_OK) { (void)cudaGetLastError(); return EMO_E_CUDA; }
        emo_walk<<<plan.walk_grid, (q.groups + 1) * 32, plan.walk_smem, st>>>(q);
        EMO_CUDA(cudaGetLastError());
    } else if (which == kIntervalFlow) {
        // the lane-stream forward kernel with the look-up inside the chain: uniform grids, F's columns in shared memory
        const FlowPlan &fp = plan.flow;
        FlowParams q = fp.pf;
        q.B = B;
        q.lvl = nullptr;
        q.ldb = 0;
        q.restore = nullptr;
        q.makespan = makespan;
        q.energy = energy;
        q.status = status;
        q.F = F;
        q.ldF = ldb;
        q.I = I;
        q.rowsF = rows;
        q.delta = delta;
        q.inv_mean = inv_mean;
        q.breaks = (const long long *)d_breaks;
        q.busy = busy;
        q.ldw = ldw;
        // Where the lanes often change the device, or an interval holds less than an entry of a lane, keeping the interval at hand costs
        // more than it saves: every entry looks its interval up.  Measured (ms, at hand / looked up): 8 devices on 18 lanes, 20 % of a lane's
        // packs on another device than the one before, 38 000 nodes x 8 192 policies 3.06 / 2.83 with 2 intervals, 5.27 / 4.69 with 200;
        // one device, 3 lanes, 2 500 packs x 16 384: 800 intervals 1.99 / 2.04, 1 600 4.46 / 4.35; 2 lanes, 250 packs: 200 0.310 /
        // 0.282 (100: 0.237 / 0.223 would pay, the line is where 5 000 nodes turn); 25 000 nodes, 100 intervals 1.43 / 2.43.
        const DevFlow &df = g->dflow;
        const bool dense = df.switches * 20 > df.packs * 3 || (int64_t)g->flow.lanes * I > df.packs;
        void (*kern)(FlowParams) = nullptr;
        if (dense) kern = fp.threads <= 512 ? emo_flow_fwd<512, true, false, true> : (fp.threads <= 768 ? emo_flow_fwd<768, true, false, true> : emo_flow_fwd<1024, true, false, true>);
        else kern = fp.threads <= 512 ? emo_flow_fwd<512, true, false> : (fp.threads <= 768 ? emo_flow_fwd<768, true, false> : emo_flow_fwd<1024, true, false>);
        if (flow_optin(kern, g) != EMO_OK) { (void)cudaGetLastError(); return EMO_E_CUDA; }
        kern<<<fp.grid_f, fp.threads, fp.smem_f, st>>>(q);
        EMO_CUDA(cudaGetLastError());
    } else {
    const Program &p = g->fwd;
    const DevProgram &d = g->dfwd;
    if (p.steps == 0) return EMO_E_UNSUPPORTED;
    LaunchShape s;
    int rc = shape_for(g, p, B, s);
    if (rc) return rc;
    const size_t brk_bytes = round_up((size_t)I * 8, 16);
    const size_t budget = g->smem_optin ? g->smem_optin : 48 * 1024;
    if (d.rec_bytes % 16) return EMO_E_UNSUPPORTED;      // a warp copies a record 16 bytes per thread
    const size_t rec_pad = round_up((size_t)d.rec_bytes, 16) + 16;      // the record and, in the last 16 bytes, the node's group
    const size_t off_rec = round_up(s.smem + brk_bytes, 16);
    const size_t off_F = off_rec + (size_t)(s.threads / 32) * 4 * rec_pad;
    if (off_F > budget) return EMO_E_UNSUPPORTED;
    const int rows_ = std::max(g->h.rows, 1);
    const size_t f_bytes = (size_t)rows_ * (size_t)I * (size_t)s.groups * 32;
    const bool stage_F = off_F + f_bytes <= budget;
    IntervalParams a;
    a.p = PassParams();
    a.p.rec = d.rec;
    a.p.rows = d.groups;
    a.p.rec_bytes = d.rec_bytes;
    a.p.steps = p.steps;
    a.p.lanes = p.lanes;
    a.p.Lp = p.Lp;
    a.p.L = g->h.L;
    a.p.slots = p.slots;
    a.p.sync = p.sync;
    a.p.groups = s.groups;
    a.p.B = B;
    a.p.makespan = makespan;
    a.p.energy = energy;
    a.F = F;
    a.ldb = ldb;
    a.I = I;
    a.breaks = d_breaks;
    a.inv_mean = inv_mean;
    a.delta = delta;
    a.busy = busy;
    a.ldw = ldw;
    a.slot_bytes = (unsigned)s.smem;
    a.off_rec = (unsigned)off_rec;
    a.rec_pad = (unsigned)rec_pad;
    a.off_F = (unsigned)off_F;
    a.stage_F = stage_F ? 1 : 0;
    a.rows = rows_;
    const size_t smem = off_F + (stage_F ? f_bytes : 0);
    void (*kern)(IntervalParams) = delta > 0 ? (stage_F ? emo_pass_intervals<true, true> : emo_pass_intervals<true, false>)
                                             : (stage_F ? emo_pass_intervals<false, true> : emo_pass_intervals<false, false>);
    if (smem > 48 * 1024) EMO_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)g->smem_optin));
    kern<<<s.grid, s.threads, smem, st>>>(a);
    EMO_CUDA(cudaGetLastError());
    }
    if (p_idle) {
        emo_idle_energy<<<(unsigned)((B + 255) / 256), 256, 0, st>>>(B, rows, I, d_breaks, F, ldb, busy, ldw, p_idle, g->h.L, makespan,
                                                                       energy, energy_idle);
        EMO_CUDA(cudaGetLastError());
    }
    if (ev1) EMO_CUDA(cudaEventRecord(ev1, st));
    return EMO_OK;
}

int emo_eval_intervals(const emo_graph *g, int64_t B, const uint8_t *F, int64_t ldb, int32_t I, const int64_t *breaks,
                       const double *p_idle, int64_t *makespan, double *energy, double *energy_idle, void *ws,
                       size_t ws_bytes, int32_t *status, uint32_t flags, void *stream)
{
    return eval_intervals(g, B, F, ldb, I, breaks, p_idle, makespan, energy, energy_idle, ws, ws_bytes, status, flags, 1, stream);
}

int emo_call_intervals(const emo_graph *g, int64_t B, int32_t I, const int64_t *breaks, uint32_t flags)
{
    if (!g || B < 0 || I < 1 || I > 4096 || !breaks) return EMO_E_INVALID_ARG;
    if (g->host_only) return EMO_E_CUDA;
    if (g->generic) return EMO_E_UNSUPPORTED;
    IntervalPlan plan;
    return interval_kernel(g, B, I, interval_length(I, breaks), flags, 1, plan);
}

// Workspace of emo_search_dp: the candidates' levels, their times and energies, and what the evaluation needs.
static void search_layout(const emo_graph *g, int32_t I, int64_t batch, int with_idle, size_t &off_T, size_t &off_E, size_t &off_ws,
                          size_t &total, int64_t &ldb)
{
    ldb = (int64_t)round_up((size_t)batch, 16);
    const size_t f_bytes = round_up((size_t)std::max(g->h.rows, 1) * (size_t)I * (size_t)ldb, 256);
    off_T = f_bytes;
    off_E = off_T + round_up((size_t)batch * 8, 256);
    off_ws = off_E + round_up((size_t)batch * 8, 256);
    size_t iv = 0;
    emo_workspace_bytes_intervals(g, batch, I, with_idle, &iv);
    total = off_ws + iv;
}

int emo_workspace_bytes_search(const emo_graph *g, int32_t I, int64_t max_batch, int with_idle, size_t *out)
{
    if (!g || !out || I < 1 || max_batch < 0) return EMO_E_INVALID_ARG;
    if (max_batch == 0) max_batch = 16384;
    size_t a, b, c, total;
    int64_t ldb;
    search_layout(g, I, max_batch, with_idle, a, b, c, total, ldb);
    *out = total;
    return EMO_OK;
}

int emo_search_dp(const emo_graph *g, int32_t I, const int64_t *breaks, const double *p_idle, int64_t T_max, int64_t bin_ns,
                  int64_t max_batch, uint8_t *F_best, int64_t *T_best, double *E_best, int64_t *n_pred, int32_t *found,
                  void *ws, size_t ws_bytes, void *stream)
{
    if (!g || I < 1 || I > 4096 || !breaks || bin_ns < 1 || max_batch < 0 || !found) return EMO_E_INVALID_ARG;
    if (g->host_only) return EMO_E_CUDA;
    if (max_batch == 0) max_batch = 16384;
    const int L = g->h.L, rows = std::max(g->h.rows, 1);
    size_t off_T, off_E, off_ws, total;
    int64_t ldb;
    search_layout(g, I, max_batch, p_idle != nullptr, off_T, off_E, off_ws, total, ldb);
    if (!ws || ws_bytes < total) return EMO_E_OOM;
    cudaStream_t st = (cudaStream_t)stream;
    uint8_t *dF = (uint8_t *)ws;
    int64_t *dT = (int64_t *)((char *)ws + off_T);
    double *dE = (double *)((char *)ws + off_E);
    void *iws = (char *)ws + off_ws;
    const size_t iws_bytes = total - off_ws;
    struct State {
        int64_t t;
        double E;
        std::vector<uint8_t> P;
    };
    int64_t calls = 0;
    *found = 0;
    // One kernel for all batches of a round: it compares their energies, and two kernels add them in different orders.  (Energies of
    // different rounds are not compared.)  The walk kernel where the rule takes it for the round's first batch: what fits it with many
    // policies fits with fewer.
    const long long delta = interval_length(I, breaks);
    bool walk = false;
    auto choose = [&](int64_t candidates) {
        IntervalPlan plan;
        walk = !g->generic && interval_kernel(g, std::min(candidates, max_batch), I, delta, 0, 1, plan) == kIntervalWalk;
    };
    try {
        std::vector<uint8_t> hF((size_t)rows * I * ldb);
        std::vector<int64_t> hT((size_t)max_batch);
        std::vector<double> hE((size_t)max_batch);
        // Pred of a chunk of candidates (policy c = cand[c], the same levels for every device row)
        auto predict = [&](const std::vector<const uint8_t *> &cand, const std::vector<std::pair<int32_t, uint8_t>> &patch) -> int {
            // (rows as long as this chunk: a round has hundreds of candidates, the workspace room for thousands)
            const int64_t nb = (int64_t)cand.size(), ld = (int64_t)round_up((size_t)nb, 16);
            for (int r = 0; r < rows; ++r)
                for (int32_t i = 0; i < I; ++i) {
                    uint8_t *dst = &hF[((size_t)r * I + i) * ld];
                    for (int64_t c = 0; c < nb; ++c) dst[c] = (patch[c].first == i) ? patch[c].second : cand[c][i];
                }
            if (cudaMemcpyAsync(dF, hF.data(), (size_t)rows * I * ld, cudaMemcpyHostToDevice, st) != cudaSuccess) return EMO_E_CUDA;
            int rc = eval_intervals(g, nb, dF, ld, I, breaks, p_idle, dT, dE, nullptr, iws, iws_bytes, nullptr, 0, walk ? 2 : 0, stream);
            if (rc) return rc;
            if (cudaMemcpyAsync(hT.data(), dT, (size_t)nb * 8, cudaMemcpyDeviceToHost, st) != cudaSuccess) return EMO_E_CUDA;
            if (cudaMemcpyAsync(hE.data(), dE, (size_t)nb * 8, cudaMemcpyDeviceToHost, st) != cudaSuccess) return EMO_E_CUDA;
            if (cudaStreamSynchronize(st) != cudaSuccess) return EMO_E_CUDA;
            calls += nb;
            return EMO_OK;
        };
        // P_0 = default level in all intervals; dp[0][t_0] = (E_0, P_0)   (Alg. 2 lines 1-3)
        std::map<int64_t, State> cur, nxt;
        {
            std::vector<uint8_t> P0((size_t)I, (uint8_t)(L - 1));
            choose(1);
            int rc = predict({P0.data()}, {{-1, 0}});
            if (rc) return rc;
            cur[hT[0] / bin_ns] = State{hT[0], hE[0], P0};
        }
        for (int32_t i = 0; i < I; ++i) {
            nxt.clear();
            choose((int64_t)cur.size() * L);
            // candidates in the order of Alg. 2: states by ascending time, levels ascending; evaluated in chunks
            std::vector<const uint8_t *> cand;
            std::vector<std::pair<int32_t, uint8_t>> patch;
            auto flush = [&]() -> int {
                if (cand.empty()) return EMO_OK;
                int rc = predict(cand, patch);
                if (rc) return rc;
                for (size_t c = 0; c < cand.size(); ++c) {
                    if (hT[c] > T_max) continue;
                    const int64_t key = hT[c] / bin_ns;
                    auto it = nxt.find(key);
                    if (it == nxt.end() || hE[c] < it->second.E) {      // strict: the first of equals stays
                        State s2{hT[c], hE[c], std::vector<uint8_t>(cand[c], cand[c] + I)};
                        s2.P[(size_t)i] = patch[c].second;
                        nxt[key] = std::move(s2);
                    }
                }
                cand.clear();
                patch.clear();
                return EMO_OK;
            };
            for (auto &kv : cur)
                for (int f = 0; f < L; ++f) {
                    cand.push_back(kv.second.P.data());
                    patch.push_back({i, (uint8_t)f});
                    if ((int64_t)cand.size() == max_batch) {
                        int rc = flush();
                        if (rc) return rc;
                    }
                }
            int rc = flush();
            if (rc) return rc;
            cur.swap(nxt);      // dp[i] is no longer needed
        }
        // (E*, P*) = the entry of dp[N] of least energy, the earliest time among equals
        const State *best = nullptr;
        for (auto &kv : cur)
            if (!best || kv.second.E < best->E) best = &kv.second;
        if (best) {
            *found = 1;
            if (F_best) std::memcpy(F_best, best->P.data(), (size_t)I);
            if (T_best) *T_best = best->t;
            if (E_best) *E_best = best->E;
        }
    } catch (const std::bad_alloc &) {
        return EMO_E_OOM;
    }
    if (n_pred) *n_pred = calls;
    return EMO_OK;
}

int emo_pack_model(int32_t n_packs, int32_t n_metrics, int32_t m, int32_t L, const double *Bmat, const double *feat,
                   const double *Tb, const double *Eb, double *x, double *T_out, double *E_out, int32_t *status, void *stream)
{
    if (n_packs < 0 || n_metrics < 1 || m < 1 || m > kModelMaxM || L < 1) return EMO_E_INVALID_ARG;
    if (n_packs == 0) return EMO_OK;
    if (!Bmat || !feat || !Tb || !Eb || !x || !T_out || !E_out) return EMO_E_INVALID_ARG;
    const size_t smem = ((size_t)n_metrics * m + 2 * (size_t)m * L) * sizeof(double);
    if (smem + (size_t)m * m * sizeof(double) > kModelMaxSmem) return EMO_E_UNSUPPORTED;
    int dev = 0, sms = 0;
    EMO_CUDA(cudaGetDevice(&dev));
    EMO_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    // with its own arrays the kernel passes what a launch has without asking (the same size in every call: concurrent callers
    // with tables of different sizes would otherwise race on the attribute)
    if (smem > 40 * 1024) EMO_CUDA(cudaFuncSetAttribute(emo_pack_model_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kModelMaxSmem));
    ModelParams p;
    p.n_packs = n_packs;
    p.n = n_metrics;
    p.m = m;
    p.L = L;
    p.B = Bmat;
    p.feat = feat;
    p.Tb = Tb;
    p.Eb = Eb;
    p.x = x;
    p.T_out = T_out;
    p.E_out = E_out;
    p.status = status;
    cudaStream_t st = (cudaStream_t)stream;
    cudaEvent_t ev0 = g_pass_events[0], ev1 = g_pass_events[1];
    if (ev0) EMO_CUDA(cudaEventRecord(ev0, st));
    const int per_block = kModelThreads / 16;
    const int blocks = std::min((n_packs + per_block - 1) / per_block, 3 * std::max(sms, 1));
    emo_pack_model_kernel<<<(unsigned)blocks, kModelThreads, smem, st>>>(p);
    EMO_CUDA(cudaGetLastError());
    if (ev1) EMO_CUDA(cudaEventRecord(ev1, st));
    return EMO_OK;
}

int emo_slack_batch(const emo_graph *g, int64_t B, const uint8_t *lvl, int64_t ldb, int64_t *ES,
                    int64_t *LS, int64_t *slack, int64_t ldo, int64_t *makespan, double *energy,
                    int64_t *slack_sum, int32_t *n_critical, int64_t *T0, double *E0, void *ws, size_t ws_bytes,
                    int32_t *status, uint32_t flags, void *stream)
{
    if (!g || B < 0) return EMO_E_INVALID_ARG;
    if (g->host_only) return EMO_E_CUDA;
    if (B == 0) return emo_eval_policies(g, 0, nullptr, 0, nullptr, nullptr, T0, E0, ws, ws_bytes, status, flags, stream);
    if (!lvl || !makespan || !energy || ldb < B) return EMO_E_INVALID_ARG;
    if ((ES || LS || slack) && ldo < B) return EMO_E_INVALID_ARG;
    cudaStream_t st = (cudaStream_t)stream;
    if (flags & EMO_F_VALIDATE) {
        int rc = launch_validate(g, B, lvl, ldb, status, st);
        if (rc) return rc;
    }
    if (g->generic)
        return launch_generic(g, B, lvl, ldb, true, ES, LS, slack, ldo, makespan, energy, slack_sum, n_critical, T0, E0, ws, ws_bytes,
                              st);
    {
        int rc = EMO_OK;
        if (slice_call(g, B, true, flags, {lvl, ldb, ES, LS, slack, ldo, makespan, energy, slack_sum, n_critical, T0, E0}, ws, ws_bytes, kSmallWs + lvl_area(g), st, rc))
            return rc;
    }
    if (spine_allowed(g, B, lvl, ldb, ldo, flags)) {
        SpinePlan fp;
        if (spine_plan(g, B, T0 || E0, true, ES || LS || slack_sum || n_critical, fp)) {
            const size_t head = kSmallWs + lvl_area(g);
            if (!ws || ws_bytes < head + fp.restore_bytes) return EMO_E_OOM;
            uint32_t *restore = (uint32_t *)((char *)ws + head);
            int rc = launch_spine_fwd(g, fp, B, lvl, ldb, restore, makespan, energy, T0, E0, status, flags, st);
            if (rc) return rc;
            return launch_spine_bwd(g, fp, B, lvl, ldb, restore, ES, LS, slack, ldo, makespan, slack_sum, n_critical, status, flags, st);
        }
    }
    if (flow_allowed(g, B, lvl, ldb, ldo, flags)) {
        FlowPlan fp;
        if (flow_plan(g, B, T0 || E0, true, fp)) {
            const size_t head = kSmallWs + lvl_area(g);
            if (!ws || ws_bytes < head + fp.restore_bytes) return EMO_E_OOM;
            uint32_t *restore = (uint32_t *)((char *)ws + head);
            int rc = launch_flow_fwd(g, fp, B, lvl, ldb, restore, makespan, energy, T0, E0, status, flags, st);
            if (rc) return rc;
            return launch_flow_bwd(g, fp, B, lvl, ldb, restore, ES, LS, slack, ldo, makespan, slack_sum, n_critical, status,
                                   flags, st);
        }
    }
    const int64_t ld_ws = (int64_t)round_up((size_t)B, 16);
    PassPlan pl;
    int rc = make_plan(g, B, T0 || E0, true, lvl, ldb, ES ? ldo : ld_ws, ldo, flags, pl);
    if (rc) return rc;
    int64_t *area = (int64_t *)((char *)ws + kSmallWs + lvl_area(g));
    int64_t *spill = nullptr, *es = ES;
    int64_t ldes = ldo;
    if (pl.staged) {
        if (!ws || ws_bytes < kSmallWs + lvl_area(g) + pl.spill_bytes) return EMO_E_OOM;
        spill = area;
    } else if (!es) {
        if (!ws || ws_bytes < kSmallWs + lvl_area(g) + (size_t)g->h.n * ld_ws * sizeof(int64_t)) return EMO_E_OOM;
        es = area;
        ldes = ld_ws;
    }
    rc = launch_pass(g, pl, false, B, lvl, ldb, es, ldes, spill, nullptr, nullptr, 0, makespan, energy, nullptr,
                     nullptr, T0, E0, status, st);
    if (rc) return rc;
    return launch_pass(g, pl, true, B, lvl, ldb, es, ldes, spill, LS, slack, ldo, makespan, energy, slack_sum,
                       n_critical, nullptr, nullptr, status, st);
}

int emo_slack(const emo_graph *g, const uint8_t *lvl_one, int64_t *ES, int64_t *LS, int64_t *slack,
              int64_t *makespan, double *energy, void *ws, size_t ws_bytes, int32_t *status, void *stream)
{
    if (!g || !makespan || !lvl_one) return EMO_E_INVALID_ARG;
    if (g->host_only) return EMO_E_CUDA;
    if (!ws || ws_bytes < g->one_bytes) return EMO_E_OOM;
    cudaStream_t st = (cudaStream_t)stream;
    double *const e1 = energy ? energy : (double *)((char *)ws + 1024);
    {
        int rc = EMO_OK;
        if (slice_call(g, 1, true, 0, {lvl_one, 1, ES, LS, slack, 1, makespan, e1, nullptr, nullptr, nullptr, nullptr}, ws, ws_bytes, kSmallWs + lvl_area(g), st, rc)) return rc;
    }
    // re-pitch the level vector to [rows][16] so that the staged kernels can be used; the
    // per-node outputs are written at pitch 1 directly
    uint8_t *lv = (uint8_t *)ws + kSmallWs;
    const size_t rows = (size_t)std::max(g->h.rows, 1);
    emo_spread_levels<<<(unsigned)((rows + 255) / 256), 256, 0, st>>>(lvl_one, lv, (int64_t)rows);
    EMO_CUDA(cudaGetLastError());
    return emo_slack_batch(g, 1, lv, 16, ES, LS, slack, 1, makespan, e1, nullptr, nullptr, nullptr, nullptr, ws, ws_bytes,
                           status, 0, stream);
}

int emo_baseline(const emo_graph *g, int64_t *T0, double *E0, void *ws, size_t ws_bytes, int32_t *status,
                 void *stream)
{
    if (!g || !T0 || !E0) return EMO_E_INVALID_ARG;
    return emo_eval_policies(g, 0, nullptr, 0, nullptr, nullptr, T0, E0, ws, ws_bytes, status, 0, stream);
}

int64_t emo_target_from_delta(int64_t T0, int64_t delta_ppm)
{
    return emo_budget(T0, delta_ppm);
}

int emo_select(int64_t B, const int64_t *makespan, const double *energy, int64_t target,
               const int64_t *target_dev, int64_t delta_ppm, int64_t *out_index, int64_t *out_T,
               double *out_E, void *ws, size_t ws_bytes, void *stream)
{
    if (B < 0 || !out_index) return EMO_E_INVALID_ARG;
    if (B > 0 && (!makespan || !energy)) return EMO_E_INVALID_ARG;
    if (!ws || ws_bytes < kSmallWs) return EMO_E_OOM;
    cudaStream_t st = (cudaStream_t)stream;
    int blocks = (int)std::max<int64_t>(1, std::min<int64_t>((B + 1023) / 1024, kSelectMaxBlocks));
    if (blocks == 1) {
        EMO_CUDA(launch_ahead(emo_select_one, 1, 256, 0, st, B, makespan, energy, target, target_dev, delta_ppm, out_index, out_T, out_E));
        return EMO_OK;
    }
    SelectPartial *part = (SelectPartial *)ws;
    EMO_CUDA(launch_ahead(emo_select_stage1, blocks, 256, 0, st, B, makespan, energy, target, target_dev, delta_ppm, part));
    EMO_CUDA(launch_ahead(emo_select_stage2, 1, 256, 0, st, blocks, (const SelectPartial *)part, makespan, out_index, out_T, out_E));
    return EMO_OK;
}

// ---- selection without any allocation --------------------------------------------------------
// Scratch for emo_select_static: the stage-1 candidates (one per block) live in this file-scope
// device array instead of a caller workspace.  Every GPU that loads the library holds these 16 KiB
// until the process exits.  In host code the array's name is only a stand-in; the device address
// comes from cudaGetSymbolAddress, looked up once per device.
static __device__ __align__(256) unsigned char emo_select_static_scratch[kSelectMaxBlocks * sizeof(SelectPartial)];
static void *g_select_static_ptr[64] = {nullptr};

int emo_select_static(int64_t B, const int64_t *makespan, const double *energy, int64_t target,
                      const int64_t *target_dev, int64_t delta_ppm, int64_t *out_index, int64_t *out_T,
                      double *out_E, void *stream)
{
    if (B < 0 || !out_index) return EMO_E_INVALID_ARG;
    if (B > EMO_SELECT_STATIC_MAX_B) return EMO_E_RANGE;
    if (B > 0 && (!makespan || !energy)) return EMO_E_INVALID_ARG;
    int dev = 0;
    EMO_CUDA(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64) return EMO_E_UNSUPPORTED;
    if (!g_select_static_ptr[dev]) {
        // first call on this device (it is the current one): resolve the array's device address
        void *ptr = nullptr;
        EMO_CUDA(cudaGetSymbolAddress(&ptr, emo_select_static_scratch));
        if (!ptr) return EMO_E_CUDA;
        g_select_static_ptr[dev] = ptr;
    }
    SelectPartial *part = (SelectPartial *)g_select_static_ptr[dev];
    cudaStream_t st = (cudaStream_t)stream;
    int blocks = (int)std::max<int64_t>(1, std::min<int64_t>((B + 1023) / 1024, kSelectMaxBlocks));
    // stage 1 overwrites the first `blocks` candidates and stage 2 reads exactly those, so nothing
    // left behind by an earlier call is ever read and nothing needs clearing
    EMO_CUDA(launch_ahead(emo_select_stage1, blocks, 256, 0, st, B, makespan, energy, target, target_dev, delta_ppm, part));
    EMO_CUDA(launch_ahead(emo_select_stage2, 1, 256, 0, st, blocks, (const SelectPartial *)part, makespan, out_index, out_T, out_E));
    return EMO_OK;
}

int emo_transpose_policies(int64_t B, int64_t rows, const uint8_t *src, int64_t lds, uint8_t *dst,
                           int64_t ldb, void *stream)
{
    if (B < 0 || rows < 0) return EMO_E_INVALID_ARG;
    if (B == 0 || rows == 0) return EMO_OK;
    if (!src || !dst || lds < rows || ldb < B) return EMO_E_INVALID_ARG;
    dim3 grid((unsigned)((rows + 31) / 32), (unsigned)std::min<int64_t>((B + 31) / 32, 65535));
    emo_transpose_u8<<<grid, dim3(32, 8), 0, (cudaStream_t)stream>>>(B, rows, src, lds, dst, ldb);
    EMO_CUDA(cudaGetLastError());
    return EMO_OK;
}

namespace {
int repack(bool pack, int bits, int64_t rows, int64_t B, uint8_t *packed, int64_t ldp, uint8_t *bytes, int64_t ldb, cudaStream_t st)
{
    if (bits < 1 || bits > 8 || rows < 0 || B < 0) return EMO_E_INVALID_ARG;
    if (rows == 0 || B == 0) return EMO_OK;
    const int64_t groups = (B + 7) / 8;
    if (!packed || !bytes || ldp < groups * bits || ldb < groups * 8 || ldb % 8 != 0 || ((uintptr_t)bytes % 8) != 0) return EMO_E_INVALID_ARG;
    const int64_t total = rows * groups;
    const int grid = (int)std::min<int64_t>((total + 255) / 256, 148 * 32);
    if (pack) emo_repack_levels<true><<<grid, 256, 0, st>>>(bits, rows, groups, packed, ldp, bytes, ldb);
    else emo_repack_levels<false><<<grid, 256, 0, st>>>(bits, rows, groups, packed, ldp, bytes, ldb);
    EMO_CUDA(cudaGetLastError());
    return EMO_OK;
}
}  // namespace

int emo_pack_levels(int bits, int64_t rows, int64_t B, const uint8_t *lvl, int64_t ldb, uint8_t *packed, int64_t ldp, void *stream)
{
    return repack(true, bits, rows, B, packed, ldp, const_cast<uint8_t *>(lvl), ldb, (cudaStream_t)stream);
}

int emo_unpack_levels(int bits, int64_t rows, int64_t B, const uint8_t *packed, int64_t ldp, uint8_t *lvl, int64_t ldb, void *stream)
{
    return repack(false, bits, rows, B, const_cast<uint8_t *>(packed), ldp, lvl, ldb, (cudaStream_t)stream);
}

// The passes, the selection and the copies of the per-policy results to the host, once the levels are on the device:
// packed in dev_packed (bits < 8: spread to dev_lvl first) or as bytes in dev_lvl (bits = 8).
// Workspace of the passes inside a host-buffer call: with the slice kernels' share where the caller's has room for it.
static size_t host_call_bytes(const emo_graph *g, int64_t B, uint32_t flags, int aligned, size_t ws_bytes)
{
    size_t need = 0;
    emo_workspace_bytes_for(g, B, 1, flags, aligned, &need);
    return ws_bytes >= need + 4 * round_up((size_t)B * 8, 256) + 256 ? need : pass_ws_bytes(g, B, 1, flags, aligned);
}

static int host_batch_tail(const emo_graph *g, int64_t B, int bits, const uint8_t *dev_packed, int64_t ld_packed, uint8_t *dev_lvl,
                           int64_t ldb, int64_t *slack_dev, int64_t ldo, int64_t delta_ppm, int64_t *makespan_host,
                           double *energy_host, int64_t *slack_sum_host, int32_t *n_critical_host, int64_t *sel_host, void *ws,
                           size_t need, uint32_t flags, cudaStream_t st)
{
    size_t per_policy = round_up((size_t)B * 8, 256);
    char *tail = (char *)ws + need;
    int64_t *d_T = (int64_t *)tail;
    double *d_E = (double *)(tail + per_policy);
    int64_t *d_ss = (int64_t *)(tail + 2 * per_policy);
    int32_t *d_nc = (int32_t *)(tail + 3 * per_policy);
    int64_t *d_sel = (int64_t *)(tail + 4 * per_policy);      // {index, T, E bits, T0, E0 bits}
    int32_t *d_status = (int32_t *)(d_sel + 8);
    EMO_CUDA(cudaMemsetAsync(d_sel, 0, 128, st));
    if (bits < 8) {
        int rcu = emo_unpack_levels(bits, g->h.rows, B, dev_packed, ld_packed, dev_lvl, ldb, (void *)st);
        if (rcu) return rcu;
    }
    int rc = emo_slack_batch(g, B, dev_lvl, ldb, nullptr, nullptr, slack_dev, ldo, d_T, d_E,
                             slack_sum_host ? d_ss : nullptr, n_critical_host ? d_nc : nullptr, d_sel + 3,
                             (double *)(d_sel + 4), ws, need, d_status, flags, st);
    if (rc) return rc;
    rc = emo_select(B, d_T, d_E, 0, d_sel + 3, delta_ppm, d_sel, d_sel + 1, (double *)(d_sel + 2), ws, need, st);
    if (rc) return rc;
    EMO_CUDA(cudaMemcpyAsync(makespan_host, d_T, (size_t)B * 8, cudaMemcpyDeviceToHost, st));
    EMO_CUDA(cudaMemcpyAsync(energy_host, d_E, (size_t)B * 8, cudaMemcpyDeviceToHost, st));
    if (slack_sum_host) EMO_CUDA(cudaMemcpyAsync(slack_sum_host, d_ss, (size_t)B * 8, cudaMemcpyDeviceToHost, st));
    if (n_critical_host) EMO_CUDA(cudaMemcpyAsync(n_critical_host, d_nc, (size_t)B * 4, cudaMemcpyDeviceToHost, st));
    int64_t tmp[10];
    EMO_CUDA(cudaMemcpyAsync(tmp, d_sel, sizeof(tmp), cudaMemcpyDeviceToHost, st));
    EMO_CUDA(cudaStreamSynchronize(st));
    sel_host[0] = tmp[0];
    sel_host[1] = tmp[1];
    sel_host[2] = tmp[2];
    sel_host[3] = tmp[3];
    int32_t stc;
    std::memcpy(&stc, &tmp[8], sizeof stc);
    return stc < 0 ? stc : EMO_OK;
}

int emo_slack_batch_host_packed(const emo_graph *g, int64_t B, int bits, const uint8_t *lvl_host, int64_t ld_host,
                                uint8_t *dev_packed, uint8_t *dev_lvl, int64_t ldb, int64_t *slack_dev, int64_t ldo,
                                int64_t delta_ppm, int64_t *makespan_host, double *energy_host, int64_t *slack_sum_host,
                                int32_t *n_critical_host, int64_t *sel_host, void *ws, size_t ws_bytes, uint32_t flags,
                                void *stream)
{
    if (!g || B <= 0 || !lvl_host || !dev_lvl || !makespan_host || !energy_host || !sel_host || ldb < B)
        return EMO_E_INVALID_ARG;
    if (bits < 1 || bits > 8 || (bits < 8 && !dev_packed)) return EMO_E_INVALID_ARG;
    if (g->host_only) return EMO_E_CUDA;
    size_t need = 0, total = 0;
    const int aligned = (ldb % 16 == 0 && aligned16(dev_lvl)) ? 1 : 0;
    need = host_call_bytes(g, B, flags, aligned, ws_bytes);
    total = need + 4 * round_up((size_t)B * 8, 256) + 256;
    // per-policy result arrays live behind the slack workspace
    if (!ws || ws_bytes < total) return EMO_E_OOM;
    cudaStream_t st = (cudaStream_t)stream;
    if (bits == 8) {
        if (ld_host != ldb) return EMO_E_INVALID_ARG;
        EMO_CUDA(cudaMemcpyAsync(dev_lvl, lvl_host, (size_t)g->h.rows * (size_t)ldb, cudaMemcpyHostToDevice, st));
    } else {
        // the levels cross the bus packed and are spread to bytes on the device
        EMO_CUDA(cudaMemcpyAsync(dev_packed, lvl_host, (size_t)g->h.rows * (size_t)ld_host, cudaMemcpyHostToDevice, st));
    }
    return host_batch_tail(g, B, bits, dev_packed, ld_host, dev_lvl, ldb, slack_dev, ldo, delta_ppm, makespan_host, energy_host,
                           slack_sum_host, n_critical_host, sel_host, ws, need, flags, st);
}

int emo_levels_prefetch(const emo_graph *g, const uint8_t *lvl_host, int64_t ld_host, uint8_t *dev_packed, void *copy_stream,
                        void *ready)
{
    if (!g || !lvl_host || !dev_packed || !ready || ld_host <= 0) return EMO_E_INVALID_ARG;
    if (g->host_only) return EMO_E_CUDA;
    cudaStream_t cs = (cudaStream_t)copy_stream;
    EMO_CUDA(cudaMemcpyAsync(dev_packed, lvl_host, (size_t)g->h.rows * (size_t)ld_host, cudaMemcpyHostToDevice, cs));
    EMO_CUDA(cudaEventRecord((cudaEvent_t)ready, cs));
    return EMO_OK;
}

int emo_slack_batch_prefetched(const emo_graph *g, int64_t B, int bits, const uint8_t *dev_packed, int64_t ld_packed, void *ready,
                               uint8_t *dev_lvl, int64_t ldb, int64_t *slack_dev, int64_t ldo, int64_t delta_ppm,
                               int64_t *makespan_host, double *energy_host, int64_t *slack_sum_host,
                               int32_t *n_critical_host, int64_t *sel_host, void *ws, size_t ws_bytes, uint32_t flags,
                               void *stream)
{
    if (!g || B <= 0 || !dev_packed || !dev_lvl || !makespan_host || !energy_host || !sel_host || ldb < B)
        return EMO_E_INVALID_ARG;
    if (bits < 1 || bits > 7) return EMO_E_INVALID_ARG;
    if (g->host_only) return EMO_E_CUDA;
    size_t need = 0, total = 0;
    const int aligned = (ldb % 16 == 0 && aligned16(dev_lvl)) ? 1 : 0;
    need = host_call_bytes(g, B, flags, aligned, ws_bytes);
    total = need + 4 * round_up((size_t)B * 8, 256) + 256;
    if (!ws || ws_bytes < total) return EMO_E_OOM;
    cudaStream_t st = (cudaStream_t)stream;
    if (ready) EMO_CUDA(cudaStreamWaitEvent(st, (cudaEvent_t)ready, 0));
    return host_batch_tail(g, B, bits, dev_packed, ld_packed, dev_lvl, ldb, slack_dev, ldo, delta_ppm, makespan_host, energy_host,
                           slack_sum_host, n_critical_host, sel_host, ws, need, flags, st);
}

int emo_slack_batch_host(const emo_graph *g, int64_t B, const uint8_t *lvl_host, int64_t ldb,
                         uint8_t *dev_lvl, int64_t *slack_dev, int64_t ldo, int64_t delta_ppm,
                         int64_t *makespan_host, double *energy_host, int64_t *slack_sum_host,
                         int32_t *n_critical_host, int64_t *sel_host, void *ws, size_t ws_bytes,
                         uint32_t flags, void *stream)
{
    return emo_slack_batch_host_packed(g, B, 8, lvl_host, ldb, nullptr, dev_lvl, ldb, slack_dev, ldo, delta_ppm, makespan_host,
                                       energy_host, slack_sum_host, n_critical_host, sel_host, ws, ws_bytes, flags, stream);
}

}  // extern "C"
