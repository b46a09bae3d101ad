// The tet corners of every vertex, in tet order (host).
#pragma once
#include <stdint.h>

#include <vector>

namespace emu {

// Index of a corner, 4 tet + its place in the tet: up to 2^30 tets have 2^32 of them.
using CornerIndex = int64_t;

struct VertexCorners {
  std::vector<CornerIndex> ptr, slot;  // vertex v: slot[ptr[v]] .. slot[ptr[v + 1] - 1]
};

inline VertexCorners vertex_corners(int64_t n, int64_t m, const int32_t* tets) {
  VertexCorners c;
  c.ptr.assign(n + 1, 0);
  c.slot.resize(4 * m);
  for (int64_t k = 0; k < 4 * m; ++k) ++c.ptr[tets[k] + 1];
  for (int64_t v = 0; v < n; ++v) c.ptr[v + 1] += c.ptr[v];
  std::vector<CornerIndex> at(c.ptr.begin(), c.ptr.end() - 1);
  for (int64_t k = 0; k < 4 * m; ++k) c.slot[at[tets[k]]++] = (CornerIndex)k;
  return c;
}

}  // namespace emu
