// Walk programs: the compiled form of a graph for time-interval policies (emo_walk.cuh).
//
// A node's level depends on its start, so a policy's nodes are evaluated one after the other by the one thread that has the policy:
// in a topological order with narrow cuts, cut into chunks, path by path inside a chunk (a node continues a path when the path's last
// node is all it waits for).  Along a path a start is the end before it.  What another path or chunk reads goes through a numbered
// slot.  Nodes outside every policy that follow each other are one (emo_contract.h).  A path is a list of items.
#pragma once
#include <cstdint>
#include <vector>

#include "emo_flow.h"

namespace emo {

constexpr int kWalkRun = 8;                      // most nodes of an item
constexpr int kWalkRows = 64;                    // nodes with a policy per chunk (their tables are brought in at once)
constexpr int kWalkNodes = 96;                   // nodes per chunk
constexpr int64_t kWalkMaxDur = 1 << 30;         // duration of a node, and of the nodes of an item together, below this: what is left of an interval
                                                 // is a signed 32-bit number

constexpr size_t kWalkShared = 227 * 1024;       // shared memory of a block

// item: word 0 nodes (bits 0..3) | flags | published slot << 16; word 1 two slots (16 bits each); word 2 fixed duration, or the nodes'
// policy row; word 3 the first node's place in the chunk's tables
constexpr uint32_t kWalkStart = 16u;             // the path begins: the later of two slots
constexpr uint32_t kWalkMore = 32u;              // ... and of what the items before it found
constexpr uint32_t kWalkFix = 64u;               // a node outside every policy
constexpr uint32_t kWalkPub = 128u;              // the end goes to a slot
constexpr uint32_t kWalkTerm = 256u;             // a node without successors: candidate for the makespan
constexpr uint32_t kWalkFresh = 512u;            // the interval is looked up (a path begins, fixed time has passed, another policy row)

struct Walk {
    bool ok = false;
    int chunks = 0, Lp = 0, slots = 0;           // slot 0 holds the time zero
    uint32_t chunk_bytes = 0, off_dur = 0, off_en = 0;      // chunk: number of items (16 bytes), items and a spare one, durations [kWalkRows][Lp], energies
    std::vector<unsigned char> blob;             // [chunks][chunk_bytes]
    double energy0 = 0.0;                        // of the nodes outside every policy
};

// Builds the walk program; ok stays false, and nothing is kept, where it does not apply (a duration too long, too many slots, chunks too long for
// a block).
void compile_walk(const HostGraph &g, const int64_t *lat, const double *energy, const GraphBounds &b, Walk &out);

}  // namespace emo
