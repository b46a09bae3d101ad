// Block-level FP64 reduction used by the per-tet kernels.
#pragma once
#include <cuda_runtime.h>

namespace emu {

// Halving butterfly of C values (a power of two, at most 64) over one warp in
// a fixed order: at each step a lane keeps half of its values and adds its
// partner's copy of that half. Lane l ends with the sums of the values
// warp_halve_first<C>(l) .. in v[0..max(C / 32, 1)). Every value's additions
// pair the lanes as a plain xor tree does (the same bits), with about C adds a
// lane instead of 5 C: on GB300 each FP64 warp instruction takes its warp 64
// cycles, whatever its lanes or its neighbours do.
template <int C, int O = 16>
__device__ __forceinline__ void warp_halve(double* v, int lane) {
  if constexpr (C >= 2) {
    constexpr int H = C / 2;
    const bool hi = (lane & O) != 0;
#pragma unroll
    for (int i = 0; i < H; ++i) {
      const double send = hi ? v[i] : v[H + i];
      const double keep = hi ? v[H + i] : v[i];
      v[i] = keep + __shfl_xor_sync(0xffffffffu, send, O);
    }
    if constexpr (O > 1) warp_halve<H, O / 2>(v, lane);
  } else {
    v[0] += __shfl_xor_sync(0xffffffffu, v[0], O);
    if constexpr (O > 1) warp_halve<1, O / 2>(v, lane);
  }
}
template <int C>
__device__ __forceinline__ int warp_halve_first(int lane) {
  if constexpr (C >= 32) return lane * (C / 32);
  return lane / (32 / C);
}
__host__ __device__ constexpr int pow2_ceil(int x) { return x <= 1 ? 1 : 2 * pow2_ceil((x + 1) / 2); }

// Sums v[0..NV) over the block (<= 256 threads) in a fixed order and writes
// the NV totals to out[0..NV). Deterministic for a fixed launch shape.
template <int NV>
__device__ __forceinline__ void block_reduce_write(double (&v)[NV], double* out) {
  constexpr int P = pow2_ceil(NV);
  __shared__ double sm[8 * P];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  double t[P];
#pragma unroll
  for (int k = 0; k < P; ++k) t[k] = k < NV ? v[k] : 0.0;
  warp_halve<P>(t, lane);
  const int first = warp_halve_first<P>(lane);
#pragma unroll
  for (int k = 0; k < (P >= 32 ? P / 32 : 1); ++k) sm[warp * P + first + k] = t[k];  // equal copies when P < 32
  __syncthreads();
  for (int k = threadIdx.x; k < NV; k += blockDim.x) {
    double x = 0.0;
    for (int w = 0; w < nw; ++w) x += sm[w * P + k];
    out[k] = x;
  }
}

// Sum of partials[b * NV + k] over b < nblk for k < NV, by a whole block of
// 256 threads: each thread takes a strided subset of the blocks, then a fixed
// tree; every k total lands in out[k] (shared or global). Deterministic.
template <int NV>
__device__ __forceinline__ void thread_sum_partials(const double* partials, int nblk, double* v) {
#pragma unroll
  for (int k = 0; k < NV; ++k) v[k] = 0.0;
  // eight strides of loads in flight at once, added in a fixed order
  constexpr int U = 8;
  const int step = blockDim.x;
  int b = threadIdx.x;
  for (; b + (U - 1) * step < nblk; b += U * step) {
    double t[U][NV];
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
      for (int k = 0; k < NV; ++k) t[u][k] = __ldcg(partials + (size_t)(b + u * step) * NV + k);
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
      for (int k = 0; k < NV; ++k) v[k] += t[u][k];
  }
  for (; b < nblk; b += step) {
#pragma unroll
    for (int k = 0; k < NV; ++k) v[k] += __ldcg(partials + (size_t)b * NV + k);
  }
}
template <int NV>
__device__ __forceinline__ void block_sum_partials(const double* partials, int nblk, double* out) {
  double v[NV];
  thread_sum_partials<NV>(partials, nblk, v);
  block_reduce_write<NV>(v, out);
  __syncthreads();
}

// True in the block that finishes last among the grid's blocks: each block
// takes a ticket after its partial sums, and the block with the last ticket
// may read every block's partials (__ldcg). One acquire-release addition by
// one thread orders them: the block barrier before it makes the block's writes
// part of the release, the one after hands the acquire on (fences by every
// thread on both sides cost 4,400 cycles, measured in the capacitance kernel).
// The caller resets *ticket to 0 from that block.
__device__ __forceinline__ bool last_block(unsigned* ticket) {
  __shared__ bool s_last;
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned t;
    asm volatile("atom.add.acq_rel.gpu.global.u32 %0, [%1], 1;" : "=r"(t) : "l"(ticket) : "memory");
    s_last = t == gridDim.x - 1;
  }
  __syncthreads();
  return s_last;
}

}  // namespace emu
