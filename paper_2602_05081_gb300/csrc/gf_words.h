// gf_words.h -- stack and queue words of the scattering renderer's traversal: an index and
// the slot (0..31) of the ray it belongs to (host and device code).
//
// Primitives are below 2^26 (gf_load_field).  Four-wide nodes may be more: there are two
// forests (by cells, by bands), and the nodes of a binary tree of c leaves at even depth are
// at most (2 c - 1) / 3 (each of them but the root is a child of one at odd depth, and
// there are c - 1 in all).  So words are unsigned, with 27 bits of index.
#pragma once
#include <stdint.h>

#ifndef GF_HD
#ifdef __CUDACC__
#define GF_HD __host__ __device__ __forceinline__
#else
#define GF_HD inline
#endif
#endif

namespace gf {

constexpr int64_t kMaxPrims = 1ll << 26;       // exclusive
constexpr int64_t kMaxNodes4 = (1ll << 27) - 1;  // exclusive: the last index is kNoWord's
constexpr uint32_t kNoWord = 0xFFFFFFFFu;

GF_HD uint32_t index_word(uint32_t index, uint32_t slot) { return index << 5 | slot; }
GF_HD uint32_t word_index(uint32_t w) { return w >> 5; }
GF_HD uint32_t word_slot(uint32_t w) { return w & 31u; }

// four-wide nodes of both forests at most: a root for each class of one primitive (57 cells,
// 8 bands) beside the nodes at even depth
constexpr int64_t max_nodes4(int64_t n) { return 2 * ((2 * n) / 3) + 64 + 8; }
static_assert(max_nodes4(kMaxPrims - 1) < kMaxNodes4, "node indices fit their words");

}  // namespace gf
