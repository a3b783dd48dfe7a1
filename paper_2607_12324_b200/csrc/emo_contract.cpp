// See emo_contract.h.
#include "emo_contract.h"

namespace emo {

void contract_forward(const HostGraph &g, const int64_t *lat, const double *energy, const GraphBounds &b, bool fixed_only, Contracted &out)
{
    out = Contracted();
    const int32_t n = g.n;
    const int L = g.L;
    // per node: live operands (the last one found), how many nodes wait for it
    std::vector<int32_t> live((size_t)n, 0), only((size_t)n, -1), waits((size_t)n, 0);
    for (int32_t v = 0; v < n; ++v)
        for (int64_t e = b.pp[v]; e < b.pp[v + 1]; ++e)
            if (b.liveF[e]) {
                ++live[v];
                only[v] = b.pc[e];
                ++waits[b.pc[e]];
            }
    // row that a node's tables depend on: -1 none; joined nodes share the first one's place
    auto row_of = [&](int32_t v) { return g.group[v] >= 0 && !(b.constant[v] && !fixed_only) ? g.group[v] : -1; };
    std::vector<int32_t> place((size_t)n, -1), row;
    std::vector<int64_t> longest;                // of the joined node (tables hold 32-bit durations)
    row.reserve((size_t)n);
    longest.reserve((size_t)n);
    for (int32_t v = 0; v < n; ++v) {
        const int32_t r = row_of(v);
        if (live[v] == 1 && waits[only[v]] == 1) {
            const int32_t p = place[only[v]];
            if ((row[p] < 0 || r < 0 || row[p] == r) && !(fixed_only && (row[p] >= 0 || r >= 0)) && longest[p] + b.dmax[v] < ((int64_t)1 << 32)) {
                place[v] = p;
                longest[p] += b.dmax[v];
                if (r >= 0) row[p] = r;
                continue;
            }
        }
        place[v] = (int32_t)row.size();
        row.push_back(r);
        longest.push_back(b.dmax[v]);
    }
    const int32_t k = (int32_t)row.size();
    out.n = k;
    out.group = row;
    out.lat.assign((size_t)k * L, 0);
    out.energy.assign((size_t)k * L, 0.0);
    // nodes are placed in the order of their first members, an edge enters there: numbered topologically
    std::vector<int32_t> first((size_t)k, -1);
    for (int32_t v = 0; v < n; ++v) {
        const int32_t p = place[v];
        if (first[p] < 0) first[p] = v;
        int64_t *const t = out.lat.data() + (size_t)p * L;
        double *const e = out.energy.data() + (size_t)p * L;
        for (int l = 0; l < L; ++l) {
            const size_t at = (size_t)v * L + (g.group[v] >= 0 ? l : 0);
            t[l] += lat[at];
            e[l] += energy[at];
        }
    }
    out.row_ptr.assign(1, 0);
    for (int32_t p = 0; p < k; ++p) {
        const int32_t v = first[p];
        for (int64_t e = b.pp[v]; e < b.pp[v + 1]; ++e)
            if (b.liveF[e]) out.col.push_back(place[b.pc[e]]);
        out.row_ptr.push_back((int64_t)out.col.size());
    }
}

}  // namespace emo
