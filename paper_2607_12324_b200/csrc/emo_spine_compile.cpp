// Back-end for spine programs (see emo_flow.h): segments, the spine's operations per direction with
// their value slots, the segment and member lists of the storing warps.
#include <algorithm>
#include <cstring>

#include "../../include/emo.h"
#include "emo_flow.h"

namespace emo {

namespace {

struct Seg {
    int32_t stage = 0, lane = 0, first = 0, count = 0, head = -1, tail = -1;
    uint32_t flags = 0;
    uint32_t acc = 0;         // word offset of the segment's sum inside the stage's sums
    int32_t idx = 0;          // index inside its stage (forward order)
    int32_t push = -1;        // restore row inside the stage, -1: the head's start follows from the lane's value
    int32_t pubF = -1, pubB = -1, readersF = 0, readersB = 0;
};

// Free list of slot numbers; slots [0, fixed) are never handed out.
struct SlotPool {
    std::vector<int32_t> free_ids;
    int32_t next = 0;
    int32_t take()
    {
        if (!free_ids.empty()) {
            const int32_t id = free_ids.back();
            free_ids.pop_back();
            return id;
        }
        return next++;
    }
    void give(int32_t id) { free_ids.push_back(id); }
};

// An operation before it has slots: where its two operands come from and what it writes.
enum class From : uint8_t { Zero, Lane, Pub, Temp, Fold };
struct Ref {
    From from = From::Zero;
    int32_t id = 0;           // lane, segment (Pub), merge operation of the stage (Temp) or reading node (Fold)
    uint32_t delta = 0;
};
struct Op {
    Ref in[2];
    int32_t seg = -1;         // the segment it completes (-1: a merge operation)
    int32_t dep[3] = {-1, -1, -1};   // operations of the same stage that come before it
    int32_t height = 1;       // longest chain of such operations that starts here
};

void note_dep(Op &o, int32_t d)
{
    if (d < 0) return;
    for (int32_t &x : o.dep) {
        if (x == d) return;
        if (x < 0) { x = d; return; }
    }
}

// Operands beyond `keep` are folded two at a time into merge operations in front of the segment's own.
template <typename Link>
void add_merges(std::vector<Op> &ops, std::vector<Ref> &refs, size_t keep, Link link)
{
    while (refs.size() > keep) {
        Op o;
        o.in[0] = refs[0];
        o.in[1] = refs[1];
        link(o);
        Ref r;
        r.from = From::Temp;
        r.id = (int32_t)ops.size();
        ops.push_back(o);
        refs.erase(refs.begin(), refs.begin() + 2);
        refs.push_back(r);               // to the back: a balanced tree
    }
}

// Order of a stage's operations in bundles of `size`: the kernel loads all operands of a bundle before it stores any
// result, so the operations of one bundle must not depend on each other.  Greedy by the length of the chain behind an
// operation; -1 = nothing to do (places of a bundle may stay empty).
std::vector<int32_t> bundle_ops(std::vector<Op> &ops, int32_t size)
{
    const int32_t m = (int32_t)ops.size();
    for (int32_t i = m - 1; i >= 0; --i)
        for (int32_t d : ops[i].dep)
            if (d >= 0) ops[d].height = std::max(ops[d].height, ops[i].height + 1);
    std::vector<int32_t> at((size_t)m, -1), order, todo((size_t)m);
    for (int32_t i = 0; i < m; ++i) todo[i] = i;
    std::stable_sort(todo.begin(), todo.end(), [&](int32_t a, int32_t b) { return ops[a].height > ops[b].height; });
    int32_t bundle = 0;
    while (!todo.empty()) {
        std::vector<int32_t> rest;
        int32_t taken = 0;
        for (int32_t i : todo) {
            bool ready = taken < size;
            for (int32_t d : ops[i].dep) ready = ready && (d < 0 || (at[d] >= 0 && at[d] < bundle));
            if (ready) {
                at[i] = bundle;
                order.push_back(i);
                ++taken;
            } else {
                rest.push_back(i);
            }
        }
        for (; taken < size; ++taken) order.push_back(-1);
        todo.swap(rest);
        ++bundle;
    }
    return order;
}

}  // namespace

int build_spine(const SpineIn &in, Spine &out, std::string &err)
{
    out = Spine();
    const int32_t n = in.n;
    const int lanes = in.lanes, K = in.K, stages = in.stages, L = in.L;
    const auto &pp = *in.pp, &sp = *in.sp;
    const auto &pc = *in.pc, &sc = *in.sc;
    const auto &liveF = *in.liveF, &liveB = *in.liveB, &constant = *in.constant;
    const auto &lbES = *in.lbES, &lbC = *in.lbC, &lbQin = *in.lbQin, &lbQ = *in.lbQ;
    const auto &step_of = *in.step_of, &lane_of = *in.lane_of, &prev = *in.prev_on_lane, &next = *in.next_on_lane, &pos_of = *in.pos_of;
    if (n == 0 || stages == 0) return EMO_OK;
    if (lanes > 255 || K > 255) return EMO_OK;
    auto stage_of = [&](int32_t v) { return step_of[v] / K; };

    // ---- what every node's live edges ask of it ---------------------------------------------------
    std::vector<int32_t> nFin((size_t)n, 0), nBout((size_t)n, 0), fold_reader((size_t)n, -1);
    std::vector<char> linkF((size_t)n, 0), linkB((size_t)n, 0), fpub((size_t)n, 0), bpub((size_t)n, 0);
    for (int32_t v = 0; v < n; ++v)
        for (int64_t e = pp[v]; e < pp[v + 1]; ++e) {
            const int32_t k = pc[e];
            const bool lane_link = prev[v] == k;
            if (liveF[e]) {
                nFin[v]++;
                if (lane_link) linkF[v] = 1;
                else fpub[k] = 1;                    // k's completion is read off its lane: k ends a segment
            }
            if (liveB[e]) {
                nBout[k]++;
                if (lane_link) {
                    linkB[v] = 1;
                } else if (fold_reader[v] < 0 && stage_of(v) >= stage_of(k) + 2) {
                    fold_reader[v] = k;              // v's tail is folded into a slot of k by the storing warps
                } else {
                    bpub[v] = 1;                     // v's tail is read off its lane: v begins a segment
                }
            }
        }
    auto invertible = [&](int32_t v) { return linkF[v] && nFin[v] == 1 && lbES[v] == lbC[prev[v]]; };
    auto pure_link = [&](int32_t v) {
        const int32_t p = prev[v];
        return p >= 0 && stage_of(p) == stage_of(v) && linkF[v] && linkB[v] && nFin[v] == 1 && nBout[p] == 1 && !fpub[p] && !bpub[v] &&
               lbES[v] == lbC[p] && lbQin[p] == lbQ[v];
    };

    // ---- segments -----------------------------------------------------------------------------------
    std::vector<int32_t> by_step((size_t)n);
    for (int32_t v = 0; v < n; ++v) by_step[v] = v;
    std::sort(by_step.begin(), by_step.end(), [&](int32_t a, int32_t b) {
        return step_of[a] != step_of[b] ? step_of[a] < step_of[b] : lane_of[a] < lane_of[b];
    });
    std::vector<Seg> segs;
    std::vector<int32_t> seg_of((size_t)n, -1);
    {
        std::vector<int32_t> open((size_t)lanes, -1);      // the lane's current segment
        for (int32_t v : by_step) {
            const int ln = lane_of[v];
            if (open[ln] >= 0 && pure_link(v) && segs[open[ln]].tail == prev[v]) {
                Seg &s = segs[open[ln]];
                s.count++;
                s.tail = v;
            } else {
                Seg s;
                s.stage = stage_of(v);
                s.lane = ln;
                s.first = pos_of[v];
                s.count = 1;
                s.head = s.tail = v;
                open[ln] = (int32_t)segs.size();
                segs.push_back(s);
            }
            seg_of[v] = open[ln];
            Seg &s = segs[open[ln]];
            bool has_energy = false;
            for (int l = 0; l < L; ++l) has_energy = has_energy || in.energy[(size_t)v * L + l] != 0.0;
            if (!constant[v]) s.flags |= kSpSeg_PreF | kSpSeg_PreB;
            else if (has_energy) s.flags |= kSpSeg_PreF;
            if (fold_reader[v] >= 0) s.flags |= kSpSeg_Fold;
        }
    }
    out.segments = (int64_t)segs.size();
    // per stage, in forward order (by the head's step, then lane): index and sum offset
    std::vector<std::vector<int32_t>> stage_segs((size_t)stages);
    for (size_t i = 0; i < segs.size(); ++i) stage_segs[segs[i].stage].push_back((int32_t)i);
    int max_segs = 0, acc_words = 0;
    for (int st = 0; st < stages; ++st) {
        auto &ss = stage_segs[st];
        std::sort(ss.begin(), ss.end(), [&](int32_t a, int32_t b) {
            const int32_t ha = segs[a].head, hb = segs[b].head;
            return step_of[ha] != step_of[hb] ? step_of[ha] < step_of[hb] : segs[a].lane < segs[b].lane;
        });
        uint32_t off = 0;
        for (size_t i = 0; i < ss.size(); ++i) {
            Seg &s = segs[ss[i]];
            s.idx = (int32_t)i;
            s.acc = off;
            off += (s.flags & kSpSeg_Fold) ? 2u : 1u;      // the sum, then X; beside it the head's tail where members are folded
        }
        max_segs = std::max(max_segs, (int)ss.size());
        acc_words = std::max(acc_words, (int)off);
    }
    out.max_segs = max_segs;
    out.acc_words = acc_words + 2;      // two scratch words behind the stage's sums (merge operations write there)
    const uint32_t scratch_acc = (uint32_t)acc_words;

    // ---- segment and member lists ---------------------------------------------------------------------
    out.n_segs.assign((size_t)stages, 0);
    out.seg.assign((size_t)stages * std::max(max_segs, 1) * kSpSegWords, 0);
    out.mem.assign((size_t)stages * lanes * K * kSpMemWords, 0);
    out.posw.assign((size_t)stages * lanes * K, 0);
    const uint32_t zero_slot = (uint32_t)lanes, dummy_slot = (uint32_t)lanes + 1u;
    auto slot_addr = [](uint32_t id) { return id * 128u; };
    if (max_segs >= 4096 || acc_words + 2 >= 65536) return EMO_OK;      // the position word has no room: no spine program
    // unused positions: no node, folds go to the slot nobody reads
    for (size_t q = 0; q < (size_t)stages * lanes * K; ++q) {
        out.mem[q * kSpMemWords + 0] = kNone;
        out.mem[q * kSpMemWords + 1] = slot_addr(dummy_slot);
        out.posw[q] = (uint32_t)(acc_words) << 16;      // sums of unused positions go to the scratch word
        out.mem[q * kSpMemWords + 3] = out.posw[q];
    }
    for (int st = 0; st < stages; ++st) {
        out.n_segs[st] = (uint32_t)stage_segs[st].size();
        for (int32_t si : stage_segs[st]) {
            const Seg &s = segs[si];
            uint32_t *w = &out.seg[((size_t)st * max_segs + s.idx) * kSpSegWords];
            const int64_t A = lbQ[s.head] + lbES[s.head];
            w[0] = (uint32_t)s.lane | ((uint32_t)s.first << 8) | ((uint32_t)s.count << 16) | (s.flags << 24);
            w[1] = s.acc * 128u;
            w[2] = (uint32_t)(uint64_t)A;
            w[3] = (uint32_t)((uint64_t)A >> 32);
            for (int32_t j = 0; j < s.count; ++j) {
                const size_t q = ((size_t)st * lanes + s.lane) * K + s.first + j;
                const uint32_t pw = (j == 0 ? kSpPos_First : 0u) | (j == s.count - 1 ? kSpPos_Last : 0u) | ((uint32_t)s.idx << 4) | (s.acc << 16);
                out.posw[q] = pw;
                out.mem[q * kSpMemWords + 3] = pw;
                out.mem[q * kSpMemWords + 4] = w[2];
                out.mem[q * kSpMemWords + 5] = w[3];
            }
        }
    }

    // ---- forward operations -----------------------------------------------------------------------------
    // fixed slots: the lanes' values, a slot that stays zero, a slot nobody reads; published values behind them
    std::vector<std::vector<uint32_t>> opsF((size_t)stages), opsB((size_t)stages);
    std::vector<std::vector<uint64_t>> pools((size_t)stages);
    out.push_base.assign((size_t)stages + 1, 0);
    out.unread_slot = dummy_slot;
    out.bundle = spine_bundle(lanes);
    {
        SlotPool pool;
        pool.next = lanes + 2;
        // readers of every published completion
        for (int32_t v = 0; v < n; ++v)
            for (int64_t e = pp[v]; e < pp[v + 1]; ++e)
                if (liveF[e] && prev[v] != pc[e]) segs[seg_of[pc[e]]].readersF++;
        std::vector<int32_t> op_of_seg(segs.size(), -1);      // operation (of its stage) that publishes the segment's value
        for (int st = 0; st < stages; ++st) {
            int32_t npush = 0;
            std::vector<Op> ops;
            std::vector<int32_t> lane_op((size_t)lanes, -1);
            auto link = [&](Op &o) {
                for (Ref &r : o.in) {
                    if (r.from == From::Pub && segs[r.id].stage == st) note_dep(o, op_of_seg[r.id]);
                    if (r.from == From::Temp) note_dep(o, r.id);
                }
            };
            for (int32_t si : stage_segs[st]) {
                Seg &s = segs[si];
                const int32_t h = s.head, t = s.tail;
                const bool terminal = sp[t + 1] == sp[t];
                const bool inv = invertible(h);
                if (!inv) s.push = npush++;
                if (inv && !(s.flags & kSpSeg_PreB) && !fpub[t] && !terminal) continue;      // the lane's value passes through unchanged
                std::vector<Ref> refs;
                // the lane's slot is always the first operand of the segment's own operation (the kernel takes the value
                // that goes to the restore list from there); a correction of 2^32 - 1 floors it to zero when the head
                // does not continue from the lane
                Ref lane_ref;
                lane_ref.from = From::Lane;
                lane_ref.id = s.lane;
                lane_ref.delta = 0xFFFFFFFFu;
                for (int64_t e = pp[h]; e < pp[h + 1]; ++e) {
                    if (!liveF[e]) continue;
                    const int32_t k = pc[e];
                    const uint32_t delta = (uint32_t)(lbES[h] - lbC[k]);
                    if (prev[h] == k) {
                        lane_ref.delta = delta;
                    } else {
                        if (segs[seg_of[k]].tail != k || !fpub[k]) { err = "internal: spine operand is not published"; return EMO_E_UNSUPPORTED; }
                        Ref r;
                        r.from = From::Pub;
                        r.id = seg_of[k];
                        r.delta = delta;
                        refs.push_back(r);
                    }
                }
                add_merges(ops, refs, 1, link);
                Op o;
                o.seg = si;
                o.in[0] = lane_ref;
                if (!refs.empty()) o.in[1] = refs[0];
                link(o);
                note_dep(o, lane_op[s.lane]);
                lane_op[s.lane] = op_of_seg[si] = (int32_t)ops.size();
                ops.push_back(o);
            }
            out.push_base[st + 1] = out.push_base[st] + npush;
            // slots are handed out in the order of execution; one that a bundle reads for the last time is free from the
            // next bundle on
            const std::vector<int32_t> order = bundle_ops(ops, out.bundle);
            std::vector<int32_t> temp_slot((size_t)ops.size(), -1), done, late;
            for (size_t i = 0; i < order.size(); ++i) {
                if (i % (size_t)out.bundle == 0) {
                    for (int32_t id : done) pool.give(id);
                    done.clear();
                }
                if (order[i] < 0) {
                    const uint32_t w8[kSpOpWordsF] = {slot_addr(zero_slot), 0u, slot_addr(zero_slot), 0u, slot_addr(dummy_slot), slot_addr(dummy_slot),
                                                      scratch_acc * 128u, kSp_NoSum};
                    opsF[st].insert(opsF[st].end(), w8, w8 + kSpOpWordsF);
                    continue;
                }
                const Op &o = ops[order[i]];
                uint32_t a[2];
                for (int k = 0; k < 2; ++k) {
                    const Ref &r = o.in[k];
                    int32_t id = (int32_t)zero_slot;
                    if (r.from == From::Lane) id = r.id;
                    if (r.from == From::Temp) done.push_back(id = temp_slot[r.id]);
                    if (r.from == From::Pub) {
                        id = segs[r.id].pubF;
                        if (id < 0) { err = "internal: spine operand has no slot"; return EMO_E_UNSUPPORTED; }
                        if (--segs[r.id].readersF == 0) done.push_back(id);
                    }
                    a[k] = slot_addr((uint32_t)id);
                }
                uint32_t fl = kSp_NoSum, acc = scratch_acc, o_lane = dummy_slot, o_pub = dummy_slot;
                if (o.seg < 0) {
                    temp_slot[order[i]] = pool.take();
                    o_pub = (uint32_t)temp_slot[order[i]];
                } else {
                    Seg &s = segs[o.seg];
                    const bool terminal = sp[s.tail + 1] == sp[s.tail];
                    if (s.flags & kSpSeg_PreB) fl = 0u;
                    if (s.push >= 0) fl |= kSp_Push | ((uint32_t)s.push << 8);
                    acc = s.acc;
                    o_lane = (uint32_t)s.lane;
                    if (terminal || (fpub[s.tail] && s.readersF > 0)) {
                        s.pubF = pool.take();
                        o_pub = (uint32_t)s.pubF;
                    }
                    if (terminal) {
                        // candidates for the makespan, taken at the end of the stage from the slots they are published in
                        fl |= kSp_Terminal;
                        pools[st].push_back((uint64_t)lbC[s.tail]);
                        out.term_slot.push_back(o_pub);
                        late.push_back((int32_t)o_pub);
                    }
                    if (s.push >= 4096 || pools[st].size() >= 4096) { err = "internal: spine stage too large"; return EMO_E_UNSUPPORTED; }
                }
                const uint32_t w8[kSpOpWordsF] = {a[0], o.in[0].delta, a[1], o.in[1].delta, slot_addr(o_lane), slot_addr(o_pub), acc * 128u, fl};
                opsF[st].insert(opsF[st].end(), w8, w8 + kSpOpWordsF);
            }
            for (int32_t id : done) pool.give(id);
            for (int32_t id : late) pool.give(id);
        }
        out.f.slots = pool.next;
    }
    out.pushes = out.push_base[stages];

    // ---- backward operations ----------------------------------------------------------------------------
    // fixed slots: the lanes' tails, zero, unread, the lanes' completion offsets, an unread one of those
    {
        // Fold slots are numbered apart from the others (tagged with the top bit until the count of the others
        // is known): a free one always holds zero, because its reader clears it.
        SlotPool pool, fpool;
        const uint32_t c_slot0 = (uint32_t)lanes + 2u, dummy_c = 2u * (uint32_t)lanes + 2u;
        const uint32_t kFoldTag = 0x80000000u;
        pool.next = 2 * lanes + 3;
        std::vector<int32_t> fold_slot((size_t)n, -1), op_of_seg(segs.size(), -1);
        for (int32_t v = 0; v < n; ++v)
            for (int64_t e = pp[v]; e < pp[v + 1]; ++e)
                if (liveB[e] && prev[v] != pc[e] && fold_reader[v] != pc[e]) segs[seg_of[v]].readersB++;
        for (int st = stages - 1; st >= 0; --st) {
            std::vector<int32_t> walk(stage_segs[st]);
            std::sort(walk.begin(), walk.end(), [&](int32_t a, int32_t b) {
                const int32_t ta = segs[a].tail, tb = segs[b].tail;
                return step_of[ta] != step_of[tb] ? step_of[ta] > step_of[tb] : segs[a].lane < segs[b].lane;
            });
            std::vector<Op> ops;
            std::vector<int32_t> lane_op((size_t)lanes, -1);
            auto link = [&](Op &o) {
                for (Ref &r : o.in) {
                    if (r.from == From::Pub && segs[r.id].stage == st) note_dep(o, op_of_seg[r.id]);
                    if (r.from == From::Temp) note_dep(o, r.id);
                }
            };
            for (int32_t si : walk) {
                Seg &s = segs[si];
                const int32_t t = s.tail;
                std::vector<Ref> refs;
                Ref lane_ref;
                bool has_lane = false, fold_seen = false;
                for (int64_t e = sp[t]; e < sp[t + 1]; ++e) {
                    const int32_t u = sc[e];
                    const int64_t ee = std::lower_bound(pc.begin() + pp[u], pc.begin() + pp[u + 1], t) - pc.begin();
                    if (!liveB[ee]) continue;
                    Ref r;
                    r.delta = (uint32_t)(lbQin[t] - lbQ[u]);
                    if (next[t] == u) {
                        // not for a merge operation: the lane's value is ordered by the segment's own operation
                        lane_ref = r;
                        lane_ref.from = From::Lane;
                        lane_ref.id = s.lane;
                        has_lane = true;
                        continue;
                    }
                    if (fold_reader[u] == t) {
                        if (fold_seen) continue;
                        fold_seen = true;
                        if (fold_slot[t] < 0) { err = "internal: spine fold slot missing"; return EMO_E_UNSUPPORTED; }
                        r.from = From::Fold;
                        r.id = t;
                        r.delta = 0;
                    } else {
                        if (segs[seg_of[u]].head != u || !bpub[u]) { err = "internal: spine tail is not published"; return EMO_E_UNSUPPORTED; }
                        r.from = From::Pub;
                        r.id = seg_of[u];
                    }
                    refs.push_back(r);
                }
                add_merges(ops, refs, has_lane ? 1 : 2, link);
                Op o;
                o.seg = si;
                int k = 0;
                if (has_lane) o.in[k++] = lane_ref;
                for (const Ref &r : refs) o.in[k++] = r;
                        link(o);
                note_dep(o, lane_op[s.lane]);
                lane_op[s.lane] = op_of_seg[si] = (int32_t)ops.size();
                ops.push_back(o);
            }
            const std::vector<int32_t> order = bundle_ops(ops, out.bundle);
            std::vector<int32_t> temp_slot((size_t)ops.size(), -1), done;
            for (size_t i = 0; i < order.size(); ++i) {
                if (i % (size_t)out.bundle == 0) {
                    for (int32_t id : done) pool.give(id);
                    done.clear();
                }
                uint32_t a[2] = {slot_addr(zero_slot), slot_addr(zero_slot)}, d[2] = {0, 0}, clear = slot_addr(dummy_slot);
                uint32_t fl = kSp_NoSum, acc = scratch_acc, qo = scratch_acc + 1u, qo_all = scratch_acc + 1u, o_lane = dummy_slot, o_pub = dummy_slot, c = dummy_c;
                if (order[i] >= 0) {
                    const Op &o = ops[order[i]];
                    for (int k = 0; k < 2; ++k) {
                        const Ref &r = o.in[k];
                        d[k] = r.delta;
                        if (r.from == From::Lane) a[k] = slot_addr((uint32_t)r.id);
                        if (r.from == From::Temp) {
                            a[k] = slot_addr((uint32_t)temp_slot[r.id]);
                            done.push_back(temp_slot[r.id]);
                        }
                        if (r.from == From::Fold) {
                            a[k] = clear = kFoldTag | slot_addr((uint32_t)fold_slot[r.id]);
                            fpool.give(fold_slot[r.id]);
                        }
                        if (r.from == From::Pub) {
                            if (segs[r.id].pubB < 0) { err = "internal: spine tail has no slot"; return EMO_E_UNSUPPORTED; }
                            a[k] = slot_addr((uint32_t)segs[r.id].pubB);
                            if (--segs[r.id].readersB == 0) done.push_back(segs[r.id].pubB);
                        }
                    }
                    if (o.seg < 0) {
                        temp_slot[order[i]] = pool.take();
                        o_pub = (uint32_t)temp_slot[order[i]];
                    } else {
                        Seg &s = segs[o.seg];
                        if (bpub[s.head] && s.readersB > 0) {
                            s.pubB = pool.take();
                            o_pub = (uint32_t)s.pubB;
                        }
                        if (s.flags & kSpSeg_PreB) fl = 0u;
                        if (s.push >= 0) fl |= kSp_Push | ((uint32_t)s.push << 8);
                        acc = s.acc;
                        if (s.flags & kSpSeg_Fold) qo = s.acc + 1u;
                        qo_all = (uint32_t)out.acc_words + (uint32_t)s.idx;
                        o_lane = (uint32_t)s.lane;
                        c = c_slot0 + (uint32_t)s.lane;
                    }
                }
                const uint32_t w12[kSpOpWordsB] = {a[0], d[0], a[1], d[1], slot_addr(o_lane), slot_addr(o_pub), acc * 128u, fl,
                                                   clear, slot_addr(c), qo * 128u, qo_all * 128u};
                opsB[st].insert(opsB[st].end(), w12, w12 + kSpOpWordsB);
            }
            for (int32_t id : done) pool.give(id);
            // the members' records.  A fold slot is taken when its first writer comes by; the stores of a stage follow the
            // stage's operations, so a slot that one of them has just cleared can be taken again here.
            for (int32_t si : walk) {
                const Seg &s = segs[si];
                int32_t u = s.head;
                for (int32_t j = 0; j < s.count; ++j, u = next[u]) {
                    uint32_t *w = &out.mem[(((size_t)st * lanes + s.lane) * K + s.first + j) * kSpMemWords];
                    w[0] = (uint32_t)u;
                    w[1] = slot_addr(dummy_slot);
                    w[6] = (uint32_t)(uint64_t)lbES[u];
                    w[7] = (uint32_t)((uint64_t)lbES[u] >> 32);
                    const int32_t r = fold_reader[u];
                    if (r >= 0) {
                        if (fold_slot[r] < 0) fold_slot[r] = fpool.take();
                        w[1] = kFoldTag | slot_addr((uint32_t)fold_slot[r]);
                        w[2] = (uint32_t)(lbQin[r] - lbQ[u]);
                    }
                }
            }
        }
        // fold slots follow the others
        const uint32_t base = (uint32_t)pool.next * 128u;
        auto fix = [&](uint32_t &w) {
            if (w & kFoldTag) w = (w & ~kFoldTag) + base;
        };
        for (auto &o : opsB)
            for (size_t i = 0; i + kSpOpWordsB <= o.size(); i += kSpOpWordsB) {
                fix(o[i + 0]);
                fix(o[i + 2]);
                fix(o[i + 8]);
            }
        for (size_t i = 0; i + kSpMemWords <= out.mem.size(); i += kSpMemWords) fix(out.mem[i + 1]);
        out.b.slots = pool.next + fpool.next;
    }

    // ---- pack --------------------------------------------------------------------------------------------
    auto pack = [&](std::vector<std::vector<uint32_t>> &src, SpineDir &d, int words) {
        size_t mx = 1;
        for (auto &o : src) mx = std::max(mx, o.size() / words);
        d.max_ops = (int)mx;
        d.n_ops.assign((size_t)stages, 0);
        d.ops.assign((size_t)stages * mx * words, 0);
        for (int st = 0; st < stages; ++st) {
            d.n_ops[st] = (uint32_t)(src[st].size() / words);
            std::copy(src[st].begin(), src[st].end(), d.ops.begin() + (size_t)st * mx * words);
        }
    };
    pack(opsF, out.f, kSpOpWordsF);
    pack(opsB, out.b, kSpOpWordsB);
    size_t mp = 1;
    for (auto &p : pools) mp = std::max(mp, p.size());
    out.max_pool = (int)mp;
    out.pool.assign((size_t)stages * mp, 0);
    for (int st = 0; st < stages; ++st) std::copy(pools[st].begin(), pools[st].end(), out.pool.begin() + (size_t)st * mp);
    out.ok = true;
    return EMO_OK;
}

}  // namespace emo
