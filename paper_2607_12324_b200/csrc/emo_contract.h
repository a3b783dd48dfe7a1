// Contraction of a graph for calls that ask for no output per node (makespan and energy only).
//
// A node whose only operand that can decide its start (static bounds, see GraphBounds) is a node that nothing else waits for
// follows it without a gap.  Where both read the same policy row, or one of them none, the two are one node whose tables are the
// sums: the makespan of every policy is the same, its energy the same sum in another order.  Edges that can never decide a maximum
// are left out.  (Nodes: 75 000 with one level per pack to 11 088, per kernel to 60 005; 38 439 of eight devices to 19 268.)
#pragma once
#include <cstdint>
#include <vector>

#include "emo_flow.h"

namespace emo {

struct Contracted {
    int32_t n = 0;
    std::vector<int64_t> row_ptr, lat;           // lat [n][L]
    std::vector<int32_t> col, group;
    std::vector<double> energy;                  // [n][L]
};

// fixed_only: only nodes outside every policy are joined, the others keep their rows (time-interval policies: a node's level depends
// on its start).
void contract_forward(const HostGraph &g, const int64_t *lat, const double *energy, const GraphBounds &b, bool fixed_only, Contracted &out);

}  // namespace emo
