// csrc/emu_corners.h: the index type holds every corner of the 2^30 tets that
// the fiber field accepts, and a small mesh's corners come out in tet order.
#include <limits>

#include "emu_corners.h"

static_assert(std::numeric_limits<emu::CornerIndex>::max() >= (int64_t(4) << 30), "4 corners of 2^30 tets");

int main() {
  const int32_t tets[12] = {0, 1, 2, 3, 3, 1, 4, 2, 5, 4, 3, 1};  // vertex 6 is in no tet
  const emu::VertexCorners c = emu::vertex_corners(7, 3, tets);
  if (c.ptr.front() != 0 || c.ptr.back() != 12) return 1;
  for (int v = 0; v < 7; ++v)
    for (auto e = c.ptr[v]; e < c.ptr[v + 1]; ++e)
      if (tets[c.slot[e]] != v || (e > c.ptr[v] && c.slot[e] <= c.slot[e - 1])) return 2;
  return c.ptr[6] == c.ptr[7] ? 0 : 3;
}
