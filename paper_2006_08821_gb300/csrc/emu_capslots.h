// Which entries of the 48 x 48 capacitance a thread of its solving block
// (k_cap) owns. Host code too, so that every (thread, slot) pair can be
// enumerated without a GPU.
#pragma once
#include <math.h>

#ifdef __CUDACC__
#define EMU_CAP_HD __host__ __device__ __forceinline__
#else
#define EMU_CAP_HD inline
#endif

namespace emu {

constexpr int kCapN = 48;                               // rows of C; B y is row 48
constexpr int kCapLow = kCapN * (kCapN + 1) / 2;        // entries of the lower triangle
constexpr int kCapSums = kCapLow + kCapN;               // and of B y
constexpr int kCapThreads = 256;
constexpr int kCapOwn = (kCapSums + kCapThreads - 1) / kCapThreads;  // entries a thread owns

// Slot ``s`` of thread ``tid`` is entry t = 1 + tid + 256 s, numbered from the
// last column backwards: column 48 - a and row 48 - b with 0 <= b <= a,
// t = a (a + 1) / 2 + b (a = 0 is unused). Slots past the last entry have
// column -1 and own nothing.
EMU_CAP_HD void cap_slot(int tid, int s, int* row, int* col) {
  const int t = 1 + tid + kCapThreads * s;
  int a = (int)((sqrtf(8.f * t + 1.f) - 1.f) * 0.5f);
  if ((a + 1) * (a + 2) / 2 <= t) ++a;
  if (a * (a + 1) / 2 > t) --a;
  *col = t <= kCapSums ? kCapN - a : -1;
  *row = t <= kCapSums ? kCapN - (t - a * (a + 1) / 2) : kCapN;
}

// Place of a slot's entry in the summed C (row-major 48 x 48) with B y behind
// it, -1 for a slot that owns nothing.
EMU_CAP_HD int cap_source(int row, int col) {
  if (col < 0) return -1;
  return row < kCapN ? row * kCapN + col : kCapN * kCapN + col;
}

}  // namespace emu
