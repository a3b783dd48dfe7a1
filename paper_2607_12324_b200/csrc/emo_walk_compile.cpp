// Compiler for walk programs (see emo_walk.h).
#include <algorithm>
#include <cstring>
#include <queue>

#include "emo_contract.h"
#include "emo_slice.h"
#include "emo_walk.h"

namespace emo {

void compile_walk(const HostGraph &g0, const int64_t *lat0, const double *energy0, const GraphBounds &b0, Walk &out)
{
    out = Walk();
    if (g0.n == 0) return;
    // the contracted graph
    Contracted c;
    contract_forward(g0, lat0, energy0, b0, true, c);
    HostGraph g;
    g.n = c.n;
    g.L = g0.L;
    g.rows = g0.rows;
    g.m = (int64_t)c.col.size();
    g.row_ptr = c.row_ptr;
    g.col = c.col;
    g.group = c.group;
    const int32_t n = g.n;
    const int L = g.L;
    GraphBounds b;
    graph_bounds(g, c.lat.data(), c.energy.data(), b);
    const std::vector<int32_t> order = narrow_order(n, b);
    for (int32_t v = 0; v < n; ++v)
        if (g.group[v] >= 0 && b.dmax[v] >= kWalkMaxDur) return;

    // items, with nodes in the place of slots
    struct Item {
        uint32_t flags = 0, fixed = 0, first = 0;
        int32_t nodes = 0, from[2] = {-1, -1}, publish = -1, row = -1;
        uint32_t slot[2] = {0, 0}, publish_slot = 0;
    };
    struct Chunk {
        std::vector<Item> items;
        std::vector<int32_t> rows;      // nodes with a policy, in walking order
    };
    std::vector<Chunk> chunks;
    std::vector<int32_t> chunk_of((size_t)n, -1), next((size_t)n, -1);
    std::vector<char> starts((size_t)n, 0);
    // paths: a node continues the path whose last node is all it waits for, inside a chunk
    {
        int32_t chunk = -1, rows = 0, nodes = 0;
        for (int32_t v : order) {
            const int32_t r = g.group[v] >= 0 ? 1 : 0;
            if (chunk < 0 || rows + r > kWalkRows || nodes == kWalkNodes) {
                ++chunk;
                rows = nodes = 0;
            }
            rows += r;
            ++nodes;
            chunk_of[v] = chunk;
            int32_t only = -1, live = 0;
            for (int64_t e = b.pp[v]; e < b.pp[v + 1]; ++e)
                if (b.liveF[e]) {
                    ++live;
                    only = b.pc[e];
                }
            if (live == 1 && chunk_of[only] == chunk && next[only] < 0) {
                next[only] = v;
            } else {
                starts[v] = 1;
            }
        }
        chunks.resize((size_t)chunk + 1);
    }
    // nodes whose end is read through a slot
    std::vector<char> published((size_t)n, 0);
    for (int32_t v = 0; v < n; ++v)
        if (starts[v])
            for (int64_t e = b.pp[v]; e < b.pp[v + 1]; ++e)
                if (b.liveF[e]) published[b.pc[e]] = 1;
    for (int32_t s : order) {
        if (!starts[s]) continue;
        Chunk &ch = chunks[(size_t)chunk_of[s]];
        std::vector<int32_t> from;
        for (int64_t e = b.pp[s]; e < b.pp[s + 1]; ++e)
            if (b.liveF[e]) from.push_back(b.pc[e]);
        for (size_t i = 0; i == 0 || i < from.size(); i += 2) {
            Item it;
            it.flags = kWalkStart | (i ? kWalkMore : 0u);
            for (int k = 0; k < 2; ++k) it.from[k] = i + (size_t)k < from.size() ? from[i + (size_t)k] : -1;
            ch.items.push_back(it);
        }
        bool fresh = true;
        int32_t row = -1;
        int64_t longest = 0;
        for (int32_t v = s; v >= 0; v = next[v]) {
            const bool term = b.sp[v + 1] == b.sp[v];
            if (g.group[v] < 0) {
                Item it;
                it.flags = kWalkFix;
                it.fixed = (uint32_t)c.lat[(size_t)v * L];
                ch.items.push_back(it);
                fresh = true;
            } else {
                Item *it = ch.items.empty() ? nullptr : &ch.items.back();
                if (fresh || g.group[v] != row || !it || it->nodes == 0 || it->nodes == kWalkRun || it->publish >= 0 || (it->flags & kWalkTerm) || longest + b.dmax[v] >= kWalkMaxDur) {
                    Item add;
                    add.flags = fresh || g.group[v] != row ? kWalkFresh : 0u;
                    add.row = g.group[v];
                    add.first = (uint32_t)ch.rows.size();
                    ch.items.push_back(add);
                    longest = 0;
                }
                ch.items.back().nodes++;
                longest += b.dmax[v];
                ch.rows.push_back(v);
                fresh = false;
                row = g.group[v];
            }
            Item &last = ch.items.back();
            if (published[v]) last.publish = v;
            if (term) last.flags |= kWalkTerm;
        }
    }

    // slots, free again after the last reader's loads
    std::vector<int64_t> last_read((size_t)n, -1);
    int64_t at = 0;
    size_t most_items = 0;
    for (const Chunk &ch : chunks) {
        most_items = std::max(most_items, ch.items.size());
        for (const Item &it : ch.items) {
            for (int32_t u : it.from)
                if (u >= 0) last_read[u] = at;
            ++at;
        }
    }
    std::priority_queue<int32_t, std::vector<int32_t>, std::greater<int32_t>> free_ids;
    std::vector<int32_t> slot((size_t)n, 0);
    int32_t slots = 1;
    at = 0;
    for (Chunk &ch : chunks)
        for (Item &it : ch.items) {
            for (int i = 0; i < 2; ++i)
                if (it.from[i] >= 0) it.slot[i] = (uint32_t)slot[it.from[i]];
            for (int i = 0; i < 2; ++i)
                if (it.from[i] >= 0 && last_read[it.from[i]] == at) free_ids.push(slot[it.from[i]]);
            if (it.publish >= 0) {
                int32_t id;
                if (!free_ids.empty()) {
                    id = free_ids.top();
                    free_ids.pop();
                } else {
                    id = slots++;
                }
                slot[it.publish] = id;
                it.publish_slot = (uint32_t)id;
            }
            ++at;
        }
    int Lp = 4;
    while (Lp < L) Lp <<= 1;
    // a block holds two chunks and a warp's slots, or no call takes the program: a node with thousands of operands makes its chunk long
    // (and all are as long), more than 128 levels make the tables of a chunk 192 KB
    const size_t off_dur = (1 + most_items + 1) * 16, off_en = off_dur + (size_t)kWalkRows * Lp * 4, bytes = off_en + (size_t)kWalkRows * Lp * 8;
    if (slots > 0xFFFF || 2 * bytes + (size_t)slots * 256 > kWalkShared) return;
    out.Lp = Lp;
    out.slots = slots;
    out.chunks = (int)chunks.size();
    out.off_dur = (uint32_t)off_dur;
    out.off_en = (uint32_t)off_en;
    out.chunk_bytes = (uint32_t)bytes;
    out.blob.assign((size_t)out.chunks * out.chunk_bytes, 0);
    for (size_t k = 0; k < chunks.size(); ++k) {
        unsigned char *const p = out.blob.data() + k * out.chunk_bytes;
        uint32_t *w = reinterpret_cast<uint32_t *>(p);
        w[0] = (uint32_t)chunks[k].items.size();
        for (const Item &it : chunks[k].items) {
            w += 4;
            w[0] = (uint32_t)it.nodes | it.flags | (it.publish >= 0 ? kWalkPub | it.publish_slot << 16 : 0u);
            w[1] = it.slot[0] | it.slot[1] << 16;
            w[2] = it.nodes ? (uint32_t)it.row : it.fixed;
            w[3] = it.first;
        }
        for (size_t r = 0; r < chunks[k].rows.size(); ++r) {
            const int32_t v = chunks[k].rows[r];
            uint32_t *const d = reinterpret_cast<uint32_t *>(p + out.off_dur) + r * (size_t)Lp;
            double *const e = reinterpret_cast<double *>(p + out.off_en) + r * (size_t)Lp;
            for (int l = 0; l < Lp; ++l) {
                d[l] = (uint32_t)c.lat[(size_t)v * L + std::min(l, L - 1)];
                e[l] = c.energy[(size_t)v * L + std::min(l, L - 1)];
            }
        }
    }
    for (int32_t v = 0; v < n; ++v)
        if (g.group[v] < 0) out.energy0 += c.energy[(size_t)v * L];
    out.ok = true;
}

}  // namespace emo
