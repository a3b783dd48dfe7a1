// Slice programs: the compiled form of a graph for calls with few policies (emo_slice.cuh).
//
// With few policies the depth of the graph is the whole cost: one after the other its nodes keep one SM busy and leave the
// rest idle.  Eq. 1 is linear in (max, +), so the graph can be cut into slices of consecutive nodes of a topological order that
// are evaluated at the same time: for every policy a slice is a matrix that takes the completion times that cross its first cut
// to those that cross its last (the longest path from each of the former to each of the latter), and the matrices are chained
// afterwards, which costs little where few values cross a cut.  Backward (tails) the same with the edges reversed.  With the
// values at the cuts known, every slice's nodes follow independently of the other slices.
//
// Inside a slice and direction the nodes form paths: a node whose only operand inside the slice is the last node of a path so far
// continues it, every other one begins a path.  Along a path values are running sums, so only where a path begins with several
// operands (or branches off) is there an operation, the maximum of its operands, each one a path's first value plus a running sum.
// They are taken two operands a step.
#pragma once
#include <cstdint>
#include <vector>

#include "emo_flow.h"

namespace emo {

constexpr int kSliceNodes = 256;                 // most nodes of a slice
constexpr int kSliceTarget = 160;                // nodes that a cut aims at
constexpr int kSliceMaxCols = 64;                // most values that cross a cut, and the time zero
constexpr int64_t kSliceMaxPath = (1 << 30) - 1; // longest path inside a slice, and along a group of them (ns): matrices are 32-bit, an absent path is negative
constexpr int kSliceScanDirect = 32;             // most slices that are chained one by one; beyond, groups of them are multiplied first

// What a slice's program says about one direction (words).
struct SliceDirHdr {
    uint32_t paths, len;                         // running sums: paths, entries (every path starts with a zero, entry 0 is one)
    uint32_t cols, outs;                         // columns: time zero, then the values that cross the cut the walk enters by; rows: (forward) the terminal
                                                 // nodes' maximum, then the values that cross the cut it leaves by
    uint32_t steps, slots1, slots2;              // steps; value slots with reuse (matrices), and one for every operation (values)
    uint32_t term;                               // forward: slot (of the second kind) that holds the terminal nodes' maximum
    uint32_t off_path, off_ops1, off_out, off_ops2;      // words from the slice's first
    uint32_t spare[4];
};
struct SliceHdr {
    uint32_t nodes, node0;                       // nodes, and the first one's place in the slice-ordered arrays
    uint32_t head, words;                        // words of header, paths and rows; all words
    uint32_t spare[4];
    SliceDirHdr dir[2];                          // forward, backward
};
constexpr int kSliceHdrWords = sizeof(SliceHdr) / 4;
constexpr int kSliceStepWords = 4;               // two operands (slot | running-sum entry << 16), the slot to write, whether it is the operation's last step

struct Slices {
    bool ok = false;
    int count = 0, cols = 0, Lp = 0;             // cols: most columns, rounded up to a multiple of four
    int group = 0, groups = 0;                   // slices per group and groups (groups = 1: chained one by one)
    std::vector<uint32_t> blob, off;             // programs; first word of every slice's (count + 1 entries)
    std::vector<uint32_t> rec;                   // [n][4] policy row (kNone: column 0), node, running-sum entry forward | backward << 16 (inclusive), slots likewise
    std::vector<uint32_t> tabT;                  // [n][Lp]
    std::vector<double> tabE;                    // [n][Lp]
};

// A topological order in which few values are alive at a time.
std::vector<int32_t> narrow_order(int32_t n, const GraphBounds &b);

// Builds the slice program; ok stays false where it does not apply (too many values cross every cut, or a path too long).
void compile_slices(const HostGraph &g, const int64_t *lat, const double *energy, const GraphBounds &b, Slices &out);

}  // namespace emo
