// One-block CSR build and orientation of small graphs (tiny.cu).
#pragma once

#include "graph.cuh"

namespace dsd {

// Where one block and the general path take the same time: G(3000, 0.0033) is
// 4 % faster on one block, 8,100 vertices with 28,000 edges took 1.41 ms
// against 1.03.
constexpr uint32_t kTinyN = 3072;    // vertices
constexpr uint32_t kTinyM = 16384;   // edge-list entries

// build_csr's result for n <= kTinyN, m <= kTinyM; *done = false (nothing kept)
// when a row with its repeats exceeds the block's buffer, or there are too many
// long ones.
dsd_status tiny_csr(dsd_graph* g, uint32_t m, const uint32_t* src, const uint32_t* dst,
                    bool* done);
// Ranks, relabelled rows and N+ starts from g->rnd; every array allocated.
dsd_status tiny_orient(dsd_graph* g);

}  // namespace dsd
