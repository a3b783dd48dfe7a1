// Compiler for slice programs (see emo_slice.h): a topological order with narrow cuts, the cuts, and per slice and direction
// paths, operations and slots.
#include <algorithm>
#include <cstdlib>
#include <queue>
#include <tuple>

#include "emo_slice.h"

namespace emo {

// A topological order in which few values are alive at a time: from the last node to the first, always the node that adds least
// to the set of nodes that placed ones still wait for, the highest-numbered among equals.  (Values alive at the best cut of every
// 64 nodes, mean / most: 250 000-node graph 5.1 / 7; in the given order, level by level, its launch nodes wait for up to 600.)
std::vector<int32_t> narrow_order(int32_t n, const GraphBounds &b)
{
    std::vector<int32_t> left((size_t)n), order((size_t)n), cur((size_t)n, 0);
    std::vector<char> ready((size_t)n, 0), live((size_t)n, 0), done((size_t)n, 0);
    using Key = std::pair<int32_t, int32_t>;      // (growth, -node)
    std::priority_queue<Key, std::vector<Key>, std::greater<Key>> heap;
    // (counted once, when the node can be placed; from then on it falls by one with every operand that begins to be waited for: nodes with
    // tens of thousands of operands are common, a host sync behind every kernel)
    auto offer = [&](int32_t v) {
        ready[v] = 1;
        cur[v] = live[v] ? -1 : 0;
        for (int64_t e = b.pp[v]; e < b.pp[v + 1]; ++e) cur[v] += live[b.pc[e]] ? 0 : 1;
        heap.push({cur[v], -v});
    };
    for (int32_t v = 0; v < n; ++v) {
        left[v] = (int32_t)(b.sp[v + 1] - b.sp[v]);
        if (left[v] == 0) offer(v);
    }
    int32_t at = n;
    while (!heap.empty()) {
        const int32_t k = heap.top().first, v = -heap.top().second;
        heap.pop();
        if (done[v] || cur[v] != k) continue;
        done[v] = 1;
        order[--at] = v;
        for (int64_t e = b.pp[v]; e < b.pp[v + 1]; ++e) {
            const int32_t u = b.pc[e];
            if (!live[u]) {
                live[u] = 1;
                for (int64_t f = b.sp[u]; f < b.sp[u + 1]; ++f)
                    if (ready[b.sc[f]] && !done[b.sc[f]]) heap.push({--cur[b.sc[f]], -b.sc[f]});
            }
            if (--left[u] == 0) offer(u);
        }
    }
    return order;
}

namespace {

struct Operand {
    int32_t slot;      // virtual slot: 0 time zero, 1 .. W the values that cross, then operations
    int32_t node;      // local node whose running sum is added (inclusive), -1: none
};
struct Op {
    std::vector<Operand> in;
    int32_t dst;
};
// The lists of one slice and direction.
struct DirLists {
    std::vector<uint32_t> paths, ops1, outs, ops2, entry, slot2;
};

// One direction of one slice.  walk: the slice's nodes in walking order; in: the nodes whose values cross the cut the walk enters by,
// out: the cut it leaves by; operands(v, f): calls f for every live operand of v; end(v): a node that nothing continues from.
template <typename Operands, typename End>
void build_dir(const std::vector<int32_t> &walk, const std::vector<int32_t> &in, const std::vector<int32_t> &out, std::vector<int32_t> &local, std::vector<int32_t> &cross,
               bool terminals, Operands operands, End end, SliceDirHdr &h, DirLists &lists)
{
    const int32_t n = (int32_t)walk.size(), W = (int32_t)in.size();
    for (int32_t i = 0; i < n; ++i) local[walk[i]] = i;
    for (int32_t j = 0; j < W; ++j) cross[in[j]] = 1 + j;

    // paths and operations
    struct Path {
        int32_t slot;
        std::vector<int32_t> nodes;
    };
    std::vector<Path> paths;
    std::vector<int32_t> path_of((size_t)n, -1);
    std::vector<Op> ops;
    int32_t next_slot = 1 + W;
    auto value_of = [&](int32_t u) -> Operand {
        return local[u] >= 0 ? Operand{paths[(size_t)path_of[local[u]]].slot, local[u]} : Operand{cross[u], -1};
    };
    for (int32_t i = 0; i < n; ++i) {
        std::vector<int32_t> from;
        operands(walk[i], [&](int32_t u) { from.push_back(u); });
        int32_t slot;
        if (from.empty()) {
            slot = 0;
        } else if (from.size() == 1 && local[from[0]] < 0) {
            slot = cross[from[0]];
        } else if (from.size() == 1 && paths[(size_t)path_of[local[from[0]]]].nodes.back() == local[from[0]]) {
            path_of[i] = path_of[local[from[0]]];
            paths[(size_t)path_of[i]].nodes.push_back(i);
            continue;
        } else {
            Op op;
            for (int32_t u : from) op.in.push_back(value_of(u));
            slot = op.dst = next_slot++;
            ops.push_back(std::move(op));
        }
        path_of[i] = (int32_t)paths.size();
        paths.push_back({slot, {i}});
    }
    Operand term{0, -1};
    if (terminals) {
        Op op;
        for (int32_t i = 0; i < n; ++i)
            if (end(walk[i])) op.in.push_back(value_of(walk[i]));
        if (!op.in.empty()) {
            term.slot = op.dst = next_slot++;
            ops.push_back(std::move(op));
        }
    }
    std::vector<Operand> outs{term};
    for (int32_t u : out) outs.push_back(value_of(u));

    // the longest paths first: they are dealt to threads in this order
    std::vector<int32_t> by_len(paths.size());
    for (size_t k = 0; k < paths.size(); ++k) by_len[k] = (int32_t)k;
    std::stable_sort(by_len.begin(), by_len.end(), [&](int32_t a, int32_t b) { return paths[(size_t)a].nodes.size() > paths[(size_t)b].nodes.size(); });
    lists.entry.assign((size_t)n, 0);
    uint32_t at = 0;
    for (int32_t k : by_len) {
        const Path &p = paths[(size_t)k];
        lists.paths.push_back(at | (uint32_t)p.nodes.size() << 16);
        for (size_t i = 0; i < p.nodes.size(); ++i) lists.entry[(size_t)p.nodes[i]] = at + 1 + (uint32_t)i;
        at += 1 + (uint32_t)p.nodes.size();
    }
    auto word = [&](const Operand &o, int32_t slot) { return (uint32_t)slot | (o.node >= 0 ? lists.entry[(size_t)o.node] : 0u) << 16; };

    // slots: of the second kind one per operation behind the one nobody reads; of the first kind free again after the last reader's
    // loads.  A step takes two operands (an odd one: the time zero, which no value is below); all but an operation's last write the
    // slot nobody reads.
    const int32_t unread = 1 + W;
    auto slot2 = [&](int32_t v) { return v <= W ? v : v + 1; };
    const int32_t never = (int32_t)ops.size();
    std::vector<int32_t> last((size_t)next_slot, -1), phys((size_t)next_slot, unread);
    for (int32_t k = 0; k < never; ++k)
        for (const Operand &o : ops[(size_t)k].in) last[(size_t)o.slot] = k;
    last[0] = never;
    for (const Operand &o : outs) last[(size_t)o.slot] = never;
    std::vector<std::vector<int32_t>> dies((size_t)never + 1);
    for (int32_t v = 0; v < next_slot; ++v)
        if (last[(size_t)v] >= 0) dies[(size_t)last[(size_t)v]].push_back(v);
    std::priority_queue<int32_t, std::vector<int32_t>, std::greater<int32_t>> free_ids;
    int32_t slots1 = unread + 1;
    for (int32_t v = 0; v <= W; ++v) {
        phys[(size_t)v] = v;
        if (last[(size_t)v] < 0) free_ids.push(v);      // a value that crosses and is only passed over here
    }
    for (int32_t k = 0; k < never; ++k) {
        const Op &op = ops[(size_t)k];
        for (size_t i = 0; i < op.in.size(); i += 2) {
            const Operand &x = op.in[i], y = i + 1 < op.in.size() ? op.in[i + 1] : Operand{0, -1};
            const uint32_t is_last = i + 2 >= op.in.size();
            for (uint32_t w : {word(x, phys[(size_t)x.slot]), word(y, phys[(size_t)y.slot]), (uint32_t)unread, is_last}) lists.ops1.push_back(w);
            for (uint32_t w : {word(x, slot2(x.slot)), word(y, slot2(y.slot)), is_last ? (uint32_t)slot2(op.dst) : (uint32_t)unread, is_last}) lists.ops2.push_back(w);
        }
        for (int32_t v : dies[(size_t)k]) free_ids.push(phys[(size_t)v]);
        if (last[(size_t)op.dst] >= 0) {
            int32_t id;
            if (!free_ids.empty()) {
                id = free_ids.top();
                free_ids.pop();
            } else {
                id = slots1++;
            }
            phys[(size_t)op.dst] = id;
            lists.ops1[lists.ops1.size() - 2] = (uint32_t)id;
        }
    }
    for (const Operand &o : outs) lists.outs.push_back(word(o, phys[(size_t)o.slot]));
    lists.slot2.assign((size_t)n, 0);
    for (int32_t i = 0; i < n; ++i) lists.slot2[(size_t)i] = (uint32_t)slot2(paths[(size_t)path_of[i]].slot);
    h.paths = (uint32_t)paths.size();
    h.len = at;
    h.cols = (uint32_t)(1 + W);
    h.outs = (uint32_t)outs.size();
    h.steps = (uint32_t)(lists.ops1.size() / kSliceStepWords);
    h.slots1 = (uint32_t)slots1;
    h.slots2 = (uint32_t)(next_slot + 1);
    h.term = (uint32_t)slot2(term.slot);
    for (int32_t i = 0; i < n; ++i) local[walk[i]] = -1;
    for (int32_t j = 0; j < W; ++j) cross[in[j]] = -1;
}

}  // namespace

void compile_slices(const HostGraph &g, const int64_t *lat, const double *energy, const GraphBounds &b, Slices &out)
{
    out = Slices();
    const int32_t n = g.n;
    if (n == 0) return;
    const std::vector<int32_t> order = narrow_order(n, b);
    std::vector<int32_t> pos((size_t)n);
    for (int32_t i = 0; i < n; ++i) pos[order[i]] = i;

    // what crosses a cut: forward the nodes before it that a node behind reads, backward the nodes behind it that one before reads
    std::vector<int32_t> until_f((size_t)n, -1), until_b((size_t)n, n);
    std::vector<int32_t> wf((size_t)n + 2, 0), wb((size_t)n + 2, 0);
    for (int32_t v = 0; v < n; ++v)
        for (int64_t e = b.pp[v]; e < b.pp[v + 1]; ++e) {
            const int32_t u = b.pc[e];
            if (b.liveF[e]) until_f[u] = std::max(until_f[u], pos[v]);
            if (b.liveB[e]) until_b[v] = std::min(until_b[v], pos[u]);
        }
    for (int32_t v = 0; v < n; ++v) {
        if (until_f[v] > pos[v]) {
            wf[(size_t)pos[v] + 1]++;
            wf[(size_t)until_f[v] + 1]--;
        }
        if (until_b[v] < pos[v]) {
            wb[(size_t)until_b[v] + 1]++;
            wb[(size_t)pos[v] + 1]--;
        }
    }
    for (int32_t i = 1; i <= n; ++i) {
        wf[i] += wf[i - 1];
        wb[i] += wb[i - 1];
    }

    // cuts: slices of about equal size, each ending where the matrices are smallest (their columns come in fours), then where
    // fewest values cross, then nearest to the size aimed at
    std::vector<int32_t> cuts{0};
    std::vector<int64_t> longest;      // longest path of every slice (ns)
    {
        std::vector<int64_t> path((size_t)n, 0);
        const int32_t want = n <= kSliceNodes ? 1 : (n + kSliceTarget - 1) / kSliceTarget, size = (n + want - 1) / want;
        while (cuts.back() < n) {
            const int32_t lo = cuts.back();
            int32_t hi = lo;      // the slice may end before any position up to hi
            while (hi < n && hi - lo < std::min(kSliceNodes, size + size / 5)) {
                const int32_t v = order[hi];
                int64_t p = 0;
                for (int64_t e = b.pp[v]; e < b.pp[v + 1]; ++e)
                    if (pos[b.pc[e]] >= lo) p = std::max(p, path[b.pc[e]]);
                path[v] = p + b.dmax[v];
                if (path[v] > kSliceMaxPath) break;
                ++hi;
            }
            if (hi == lo) return;
            int32_t best = hi;
            if (hi < n) {
                auto score = [&](int32_t c) { return std::make_tuple((std::max(wf[c], wb[c]) + 4) / 4, wf[c] + wb[c], std::abs(c - lo - size)); };
                auto search = [&](int32_t from) {
                    for (int32_t c = lo + std::max(1, from); c < hi; ++c)
                        if (score(c) < score(best)) best = c;
                };
                search(size * 7 / 10);
                if (std::get<0>(score(best)) > 2) search(size / 3);
            }
            cuts.push_back(best);
            int64_t p = 0;
            for (int32_t i = lo; i < best; ++i) p = std::max(p, path[order[i]]);
            longest.push_back(p);
        }
    }
    const int32_t C = (int32_t)cuts.size() - 1;
    int32_t most = 0;
    for (int32_t c = 1; c < C; ++c) most = std::max(most, std::max(wf[cuts[c]], wb[cuts[c]]));
    if (most + 1 > kSliceMaxCols) return;

    int Lp = 4;
    while (Lp < g.L) Lp <<= 1;
    out.Lp = Lp;
    out.count = C;
    out.cols = (most + 1 + 3) / 4 * 4;
    out.groups = 1;
    out.group = C;
    if (C > kSliceScanDirect) {
        // about as many groups as slices in each; fewer slices where their longest paths would not fit 32 bits
        while ((int64_t)out.groups * out.groups < C) ++out.groups;
        out.group = (C + out.groups - 1) / out.groups;
        auto fits = [&](int32_t k) {
            for (int32_t c = 0; c < C; c += k) {
                int64_t p = 0;
                for (int32_t i = c; i < std::min(C, c + k); ++i) p += longest[(size_t)i];
                if (p > kSliceMaxPath) return false;
            }
            return true;
        };
        while (out.group > 1 && !fits(out.group)) out.group = (out.group + 1) / 2;
        out.groups = (C + out.group - 1) / out.group;
    }
    // the values that cross each cut
    std::vector<std::vector<int32_t>> cross_f((size_t)C + 1), cross_b((size_t)C + 1);
    for (int32_t i = 0; i < n; ++i) {
        const int32_t v = order[i];
        for (auto it = std::upper_bound(cuts.begin(), cuts.end(), i); it != cuts.end() && *it <= until_f[v]; ++it)
            cross_f[(size_t)(it - cuts.begin())].push_back(v);
        if (until_b[v] < i)
            for (auto it = std::upper_bound(cuts.begin(), cuts.end(), until_b[v]); it != cuts.end() && *it <= i; ++it)
                cross_b[(size_t)(it - cuts.begin())].push_back(v);
    }

    out.rec.assign((size_t)n * 4, 0);
    out.tabT.assign((size_t)n * Lp, 0);
    out.tabE.assign((size_t)n * Lp, 0.0);
    std::vector<int32_t> local((size_t)n, -1), cross((size_t)n, -1);
    out.off.assign(1, 0);
    for (int32_t c = 0; c < C; ++c) {
        const int32_t lo = cuts[c], hi = cuts[c + 1];
        std::vector<int32_t> walk(order.begin() + lo, order.begin() + hi), back(walk.rbegin(), walk.rend());
        SliceHdr h = {};
        h.nodes = (uint32_t)(hi - lo);
        h.node0 = (uint32_t)lo;
        DirLists lists[2];
        build_dir(walk, cross_f[c], cross_f[c + 1], local, cross, true,
                  [&](int32_t v, auto f) {
                      for (int64_t e = b.pp[v]; e < b.pp[v + 1]; ++e)
                          if (b.liveF[e]) f(b.pc[e]);
                  },
                  [&](int32_t v) { return b.sp[v + 1] == b.sp[v]; }, h.dir[0], lists[0]);
        build_dir(back, cross_b[c + 1], cross_b[c], local, cross, false,
                  [&](int32_t v, auto f) {
                      for (int64_t s = b.sp[v]; s < b.sp[v + 1]; ++s)
                          if (b.liveB[b.se[s]]) f(b.sc[s]);
                  },
                  [](int32_t) { return false; }, h.dir[1], lists[1]);
        // the words of the slice
        std::vector<uint32_t> w((size_t)kSliceHdrWords, 0);
        auto put = [&](const std::vector<uint32_t> &x) {
            const uint32_t at = (uint32_t)w.size();
            w.insert(w.end(), x.begin(), x.end());
            while (w.size() % 4) w.push_back(0);
            return at;
        };
        for (int d = 0; d < 2; ++d) h.dir[d].off_path = put(lists[d].paths);
        for (int d = 0; d < 2; ++d) h.dir[d].off_out = put(lists[d].outs);
        h.head = (uint32_t)w.size();
        // (behind each list a spare step: the next one is read ahead)
        for (int d = 0; d < 2; ++d) {
            h.dir[d].off_ops1 = put(lists[d].ops1);
            w.resize(w.size() + kSliceStepWords, 0);
        }
        for (int d = 0; d < 2; ++d) {
            h.dir[d].off_ops2 = put(lists[d].ops2);
            w.resize(w.size() + kSliceStepWords, 0);
        }
        h.words = (uint32_t)w.size();
        std::copy((const uint32_t *)&h, (const uint32_t *)&h + kSliceHdrWords, w.begin());
        out.blob.insert(out.blob.end(), w.begin(), w.end());
        out.off.push_back((uint32_t)out.blob.size());
        for (int32_t i = lo; i < hi; ++i) {
            const int32_t v = order[i], fi = i - lo, bi = hi - 1 - i;
            uint32_t *r = out.rec.data() + (size_t)i * 4;
            r[0] = (g.group[v] >= 0 && !b.constant[v]) ? (uint32_t)g.group[v] : kNone;
            r[1] = (uint32_t)v;
            r[2] = lists[0].entry[fi] | lists[1].entry[bi] << 16;
            r[3] = lists[0].slot2[fi] | lists[1].slot2[bi] << 16;
            for (int l = 0; l < Lp; ++l) {
                const int s = g.group[v] >= 0 ? std::min(l, g.L - 1) : 0;
                out.tabT[(size_t)i * Lp + l] = (uint32_t)lat[(size_t)v * g.L + s];
                out.tabE[(size_t)i * Lp + l] = energy[(size_t)v * g.L + s];
            }
        }
    }
    out.ok = true;
}

}  // namespace emo
