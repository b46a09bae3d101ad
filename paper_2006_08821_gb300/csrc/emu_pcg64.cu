// FP64 conjugate gradient of the coupling solve (Eq. 4, three right-hand
// sides) with every row's state on chip: the FP64 path's dq solves and exact
// re-solves, the mixed path's solves with bones, the allocation-free solve
// and the fiber field.
//
// The iteration is the generic kernel's (pcg_kernel in emu_pcg.cu:
// Chronopoulos-Gear CG, Jacobi plus the additive coarse space). What bounds it
// on these systems (400 to 50,000 rows) is latency: two grid barriers, one L2
// gather and one sum over the blocks per iteration, and the FP64 pipe, which
// issues two FMAs per cycle and SM. So:
//   * a warp owns one column of 32 rows (three warps per 32 rows), so a row's
//     chains are 16 products long, a warp's reduction carries 19 values
//     instead of 57, and no lane idles;
//   * x, r, p, s, u, w stay in registers; the matrix (16 entries per row) and
//     the coarse rows stay in shared memory, one copy for the three columns;
//     only u goes through L2;
//   * the coarse basis comes as Phi' = Phi T with T T^T = E^-1, so
//     M = D^-1 + Phi' Phi'^T needs no 16 x 16 product between the reduction
//     and the next u;
//   * as few as 32 rows per block while a block per SM suffices: the FP64 work
//     of a row (about 165 FMAs per iteration) is what more SMs share, and the
//     barrier costs little more with 152 blocks than with 5. Rows per block
//     grow in steps of 32 once n exceeds 32 per SM (up to 320);
//   * the barrier is a release-add and an acquire poll on one counter that
//     the last block to leave zeroes, so no memset precedes a launch;
//   * one division on the path from the sums to alpha: with den the last
//     denominator, beta g / alpha = beta^2 den.
//   * a lane sums one mode of Phi'^T w over half of its warp's rows (17 FP64
//     instructions; 16 products and a butterfly are 32), products run in one
//     chain and one reciprocal serves alpha and the next beta: an FP64
//     instruction holds its warp 64 cycles whatever its lanes or its
//     neighbours do, so a warp's instruction count is its time.
// Measured on one GB300 against the generic kernel: coupling solve of 19,833
// rows 4.83 -> 1.74 ms; an iteration at 425 rows 28 -> 6.8 us, at 692 rows (the
// arm's 45 an iteration of Newton) 23 -> 7.5 us, at 1,485 rows 28 -> 8.5 us.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <mutex>

#include "emu_internal.h"
#include "emu_math.cuh"
#include "emu_pcg.h"
#include "emu_reduce.cuh"

namespace emu {

namespace {

constexpr int NR = 3;
constexpr int kEll = 16;        // entries of a matrix row held in shared memory
constexpr int kRed = 20;        // values a warp reduces: gamma, delta, rr, bb, 16 modes
constexpr int kPart = 64;       // doubles per block in the partial sums
constexpr int kMaxRows = 320;   // rows per block at most (960 threads)
constexpr int kNV = 12 + NR * kModes;  // gamma, delta, rr, bb (3 columns each), Phi'^T w

__device__ __forceinline__ void red_release_add(unsigned* p, unsigned v) {
  asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ unsigned ld_acquire(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// Grid barrier on bar->v_count (arrivals of the launch so far). Bounded: a
// wait that runs out raises v_err, every other waiter sees it and leaves.
__device__ __forceinline__ bool vbar(GridBarrier* bar, unsigned& epoch, int* s_flag, unsigned long long wait_ns) {
  __syncthreads();
  epoch += 1u;
  if (threadIdx.x == 0) {
    red_release_add(&bar->v_count, 1u);
    const unsigned target = gridDim.x * epoch;
    int bad = 0;
    unsigned long long spins = 0, t0 = 0;
    while (ld_acquire(&bar->v_count) < target) {
      ++spins;
      if ((spins & 63u) == 0u) {
        if (*((volatile unsigned*)&bar->v_err)) {
          bad = 1;
          break;
        }
        const unsigned long long now = global_ns();
        if (t0 == 0) t0 = now;
        if (now - t0 > wait_ns || spins > kWaitSpinCap) {
          bad = 1;
          atomicExch(&bar->v_err, 1u);
          break;
        }
      }
    }
    *s_flag = bad;
  }
  __syncthreads();
  return *s_flag == 0;
}

// The last block to leave zeroes the words for the next launch.
__device__ __forceinline__ void vbar_exit(GridBarrier* bar) {
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    if (atomicAdd(&bar->v_done, 1u) + 1u == gridDim.x) {
      atomicExch(&bar->v_count, 0u);
      atomicExch(&bar->v_err, 0u);
      atomicExch(&bar->v_done, 0u);
    }
  }
}

}  // namespace

// blockDim.x = max(256, 3 rows); warp w < 3 rows / 32 owns column w % 3 of
// the rows 32 (w / 3) .. + 31 of the block; further warps help with the sums.
template <int MAXT, bool COARSE>
__global__ void __launch_bounds__(MAXT, 1) pcg64_kernel(PcgArgsT<double> a, int rows) {
  constexpr int NC = COARSE ? kModes : 0;
  __shared__ double s_red[(kMaxRows / 32) * NR * kRed];
  __shared__ double s_grp[16 * kPart];
  __shared__ double s_rho[NR * kModes], s_sig[NR * kModes];
  __shared__ double s_al[NR], s_be[NR];
  __shared__ int s_act[NR], s_zero[NR];
  __shared__ int s_flag;
  extern __shared__ double dyn[];
  double* sVal = dyn;                        // [kEll][rows]
  double* sPhi = sVal + kEll * rows;         // [16][rows + 1] when COARSE
  const int ps = rows + 1;                   // its stride: sixteen modes of a row in sixteen banks
  double* sW = sPhi + NC * ps;               // [warp][32] when COARSE
  int32_t* sCol = reinterpret_cast<int32_t*>(sW + (COARSE ? NR * rows : 0));  // [kEll][rows]
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int G = gridDim.x;
  const int64_t n = a.n;
  const int64_t r0 = (int64_t)blockIdx.x * rows;
  const int nrow = (int)(n - r0 < rows ? n - r0 : rows);
  const int grp = warp / NR, j = warp % NR;  // row group and column of this warp
  const int lr = grp * 32 + lane;            // row of this thread in the block
  const bool data = grp * 32 < rows;         // a warp with rows
  const bool own = data && lr < nrow;
  const int64_t v = r0 + (own ? lr : 0);
  unsigned epoch = 0;
  double* __restrict__ ug = a.u;  // [3][n]
  double* __restrict__ part = a.partials;

  int cnt = 0;
  int32_t e0 = 0, e1 = 0;
  if (own) {
    e0 = __ldg(a.rowptr + v);
    e1 = __ldg(a.rowptr + v + 1);
    cnt = e1 - e0;
  }
  // the three warps of a row group fill its matrix entries and coarse rows
  if (data) {
    for (int t = j; t < kEll; t += NR) {
      sVal[t * rows + lr] = own && t < cnt ? __ldg(a.val + e0 + t) : 0.0;
      sCol[t * rows + lr] = own && t < cnt ? __ldg(a.col + e0 + t) : (int32_t)v;
    }
    if constexpr (COARSE)
      for (int m = j; m < kModes; m += NR) sPhi[m * ps + lr] = own ? __ldg(a.phit + (size_t)m * n + v) : 0.0;
  }
  const double di = own ? __ldg(a.dinv + v) : 0.0;
  const double bv = own ? a.b[v * NR + j] : 0.0;
  double x = own ? a.x[v * NR + j] : 0.0;
  __syncthreads();

  // one entry of A z, z element c at z[c * stride + j * plane]
  auto spmv = [&](const double* z, int64_t stride, int64_t plane) -> double {
    if (!own) return 0.0;
    const double* zj = z + j * plane;
    double acc = 0.0;  // one chain: an FP64 instruction occupies its warp as long as it takes
    constexpr int GW = MAXT > 512 ? 8 : 16;  // gathers in flight
#pragma unroll
    for (int t0 = 0; t0 < kEll; t0 += GW) {
      double zz[GW];
#pragma unroll
      for (int t = 0; t < GW; ++t) zz[t] = t0 + t < cnt ? __ldcg(zj + sCol[(t0 + t) * rows + lr] * stride) : 0.0;
#pragma unroll
      for (int t = 0; t < GW; ++t) acc = fma(sVal[(t0 + t) * rows + lr], zz[t], acc);
    }
    for (int32_t e = e0 + kEll; e < e1; e += 4) {  // long rows
      double av[4], zz[4];
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        const bool on = e + t < e1;
        av[t] = on ? __ldg(a.val + e + t) : 0.0;
        zz[t] = on ? __ldcg(zj + __ldg(a.col + e + t) * stride) : 0.0;
      }
#pragma unroll
      for (int t = 0; t < 4; ++t) acc = fma(av[t], zz[t], acc);
    }
    return acc;
  };
  // u = D^-1 r + Phi' rho
  auto precond = [&](double r) -> double {
    double acc = di * r;
    if constexpr (COARSE) {
      if (data) {
#pragma unroll
        for (int m = 0; m < kModes; ++m) acc = fma(sPhi[m * ps + lr], s_rho[j * kModes + m], acc);
      }
    }
    return acc;
  };
  // block sums of d4 (gamma, delta, rr, bb of this thread) and Phi'^T y, written as this block's partials
  auto reduce = [&](const double (&d4)[4], double y) {
    if (data) {
      double t4[4] = {d4[0], d4[1], d4[2], d4[3]};
      warp_halve<4>(t4, lane);
      if ((lane & 7) == 0) s_red[warp * kRed + (lane >> 3)] = t4[0];
      if constexpr (COARSE) {
        // mode lane % 16 over half of the warp's rows in each half of the warp:
        // 17 FP64 instructions (16 products and a halving butterfly are 32)
        double* sw = sW + warp * 32;
        sw[lane] = y;
        __syncwarp();
        const double* ph = sPhi + (lane & 15) * ps + grp * 32 + (lane & 16);
        const double* yw = sw + (lane & 16);
        double t = 0.0;
#pragma unroll
        for (int q = 0; q < 16; ++q) t = fma(ph[q], yw[q], t);
        t += __shfl_xor_sync(0xffffffffu, t, 16);
        if (lane < 16) s_red[warp * kRed + 4 + lane] = t;
        __syncwarp();
      }
    }
    __syncthreads();
    if (tid < 12 + NR * NC) {
      // value q < 12: item q / 3 of column q % 3; then mode (q - 12) % 16 of column (q - 12) / 16
      const int jj = tid < 12 ? tid % NR : (tid - 12) / kModes;
      const int item = tid < 12 ? tid / NR : 4 + (tid - 12) % kModes;
      double t = 0.0;
      for (int g = 0; g * 32 < rows; ++g) t += s_red[(g * NR + jj) * kRed + item];
      __stcg(part + (size_t)blockIdx.x * kPart + tid, t);
    }
  };
  // sum over the blocks in a fixed order: groups of 64 threads take every
  // NG-th block, eight loads in flight; thread k < kNV returns value k
  auto gather_sums = [&]() -> double {
    const int k = tid & (kPart - 1), g = tid / kPart, NG = (int)blockDim.x / kPart;
    if (k < 12 + NR * NC && g < NG) {
      double t = 0.0;
      for (int b = g; b < G; b += 8 * NG) {
        double l[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) l[q] = b + q * NG < G ? __ldcg(part + (size_t)(b + q * NG) * kPart + k) : 0.0;
#pragma unroll
        for (int q = 0; q < 8; ++q)
          if (b + q * NG < G) t += l[q];
      }
      s_grp[g * kPart + k] = t;
    }
    __syncthreads();
    double t = 0.0;
    if (tid < kPart)
      for (int gg = 0; gg < NG; ++gg) t += s_grp[gg * kPart + tid];
    return t;
  };

  // ---- r = b - A x (x in place: it is written back only after two barriers)
  double r = bv - spmv(a.x, NR, 1);
  if (!own) r = 0.0;
  if constexpr (COARSE) {  // rho = Phi'^T r
    const double z4[4] = {0.0, 0.0, 0.0, 0.0};
    reduce(z4, r);
    if (!vbar(a.bar, epoch, &s_flag, a.wait_ns)) goto timeout;
    const double t = gather_sums();
    if (tid >= 12 && tid < kNV) s_rho[tid - 12] = t;
    __syncthreads();
  }
  {
    double u = precond(r);
    if (own) __stcg(ug + j * n + v, u);
    if (!vbar(a.bar, epoch, &s_flag, a.wait_ns)) goto timeout;
    double w = spmv(ug, 1, n);
    {
      const double d4[4] = {r * u, w * u, r * r, bv * bv};
      reduce(d4, w);
    }
    if (!vbar(a.bar, epoch, &s_flag, a.wait_ns)) goto timeout;
    // scalars of column l in lane l of warp 0
    double sden = 0.0, sig_ = 0.0, sthr = 0.0, sbb = 0.0, srr = 0.0, sal = 0.0;
    int sact = 0;
    double t = gather_sums();
    if (warp == 0) {
      const double g = t, dl = __shfl_sync(0xffffffffu, t, (lane + 3) & 31), rr = __shfl_sync(0xffffffffu, t, (lane + 6) & 31),
                   bb = __shfl_sync(0xffffffffu, t, (lane + 9) & 31);
      if (lane < NR) {
        sbb = bb;
        srr = rr;
        sthr = a.tol * a.tol * bb;
        sden = dl;
        sig_ = 1.0 / g;
        sact = (rr <= sthr || !(dl > 0.0)) ? 0 : 1;
        sal = sact ? g / dl : 0.0;
        s_al[lane] = sal;
        s_be[lane] = 0.0;
        s_act[lane] = sact;
        s_zero[lane] = bb == 0.0;
      }
    }
    __syncthreads();
    if (COARSE && tid >= 12 && tid < kNV) {
      const int q = tid - 12;
      s_sig[q] = t;
      if (s_act[q / kModes]) s_rho[q] -= s_al[q / kModes] * t;
    }
    __syncthreads();
    double p = u, s = w;
    if (s_zero[j]) x = 0.0;  // zero right-hand side: x = 0 exactly
    int it = 0;
    bool all_done = !(s_act[0] || s_act[1] || s_act[2]);
    while (!all_done && it < a.max_iter) {
      ++it;
      if (s_act[j]) {
        const double al = s_al[j];
        x = fma(al, p, x);
        r = fma(-al, s, r);
      }
      u = precond(r);
      if (own) __stcg(ug + j * n + v, u);
      if (!vbar(a.bar, epoch, &s_flag, a.wait_ns)) goto timeout;
      w = spmv(ug, 1, n);
      {
        const double d4[4] = {r * u, w * u, r * r, 0.0};
        reduce(d4, w);
      }
      if (!vbar(a.bar, epoch, &s_flag, a.wait_ns)) goto timeout;
      t = gather_sums();
      if (warp == 0) {
        const double g = t, dl = __shfl_sync(0xffffffffu, t, (lane + 3) & 31),
                     rr = __shfl_sync(0xffffffffu, t, (lane + 6) & 31);
        const double be = g * sig_;
        const double den = fma(-be, be * sden, dl);
        // 1 / den in lanes 0 .. 2 and 1 / g, for the next iteration, in 3 .. 5
        const double gs = __shfl_sync(0xffffffffu, g, (lane + 29) & 31);
        const double inv = inv_n(lane < NR ? den : gs);
        const double al = g * inv, ig = __shfl_sync(0xffffffffu, inv, (lane + NR) & 31);
        if (lane < NR && sact) {
          srr = rr;
          // rr <= sthr on the bits (both are sums of squares)
          if (__double_as_longlong(rr) <= __double_as_longlong(sthr) || !positive_n(den)) {
            sact = 0;  // converged, or breakdown: stop this column
            s_act[lane] = 0;
          } else {
            s_be[lane] = be;
            s_al[lane] = al;
            sig_ = ig;
            sden = den;
          }
        }
      }
      __syncthreads();
      if (COARSE && tid >= 12 && tid < kNV) {  // sigma = Phi'^T w + beta sigma, rho -= alpha sigma
        const int q = tid - 12, c = q / kModes;
        if (s_act[c]) {
          const double sg2 = fma(s_be[c], s_sig[q], t);
          s_sig[q] = sg2;
          s_rho[q] -= s_al[c] * sg2;
        }
      }
      if (s_act[j]) {
        const double be = s_be[j];
        p = fma(be, p, u);
        s = fma(be, s, w);
      }
      all_done = !(s_act[0] || s_act[1] || s_act[2]);
      __syncthreads();
    }
    if (own) a.x[v * NR + j] = x;
    if (blockIdx.x == 0 && warp == 0) {
      if (lane == 0) {
        if (a.iters_out) atomicAdd(a.iters_out, it);
        if (a.fail_out && !all_done) atomicExch(a.fail_out, 1);
        if (a.last_iters) *a.last_iters = it;
      }
      if (lane < NR && a.relres_out) a.relres_out[lane] = sbb > 0.0 ? sqrt(srr / sbb) : 0.0;
    }
  }
  vbar_exit(a.bar);
  return;
timeout:
  if (tid == 0 && a.timeout_out) atomicExch(a.timeout_out, 1);
  vbar_exit(a.bar);
}

namespace {
size_t pcg64_smem(int rows, bool coarse) {
  return (size_t)rows * (8 * kEll + 4 * kEll + (coarse ? 8 * kModes + 8 * NR : 0)) + (coarse ? 8 * kModes : 0);
}

template <int MAXT, bool C>
cudaError_t launch64(const PcgArgsT<double>& args, int rows, int grid, int threads, cudaStream_t st) {
  // Every shape of an instantiation within one limit, raised once per device.
  // (Static and dynamic bytes together decide: 13 to 14 KB of static arrays
  // pass the default 48 KB with 192 rows without a coarse space already.)
  {
    static bool set[64] = {false};
    static std::mutex mu;
    std::lock_guard<std::mutex> lock(mu);
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    if (!set[dev]) {
      e = cudaFuncSetAttribute(pcg64_kernel<MAXT, C>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               (int)pcg64_smem(MAXT / NR, C));
      if (e != cudaSuccess) return e;
      set[dev] = true;
    }
  }
  const size_t smem = pcg64_smem(rows, C);
  PcgArgsT<double> a = args;
  int r = rows;
  void* params[] = {(void*)&a, (void*)&r};
  return cudaLaunchCooperativeKernel((const void*)pcg64_kernel<MAXT, C>, dim3(grid), dim3(threads), params, smem, st);
}

template <bool C> cudaError_t pick64(const PcgArgsT<double>& a, int rows, int grid, cudaStream_t st) {
  const int threads = std::max(256, NR * rows);
  if (threads <= 288) return launch64<288, C>(a, rows, grid, threads, st);
  if (threads <= 480) return launch64<480, C>(a, rows, grid, threads, st);
  return launch64<960, C>(a, rows, grid, threads, st);
}
}  // namespace

// ------------------------------------------------- sixteen right-hand sides --
// The same CG without a coarse space for 16 columns: the subspace iteration of
// the low-rank basis (Eq. 9) and the joints' responses, at set-up. The generic
// kernel gives a thread one row and 16 columns, about 550 FP64 instructions an
// iteration at 64 cycles each (70 us at 1,485 rows, 45 of the 50 ms of a
// 6,080-tet handle's set-up). Here a warp owns one column of 32 rows and a
// block CPB columns of 128 rows, so the columns of a small system spread over
// the SMs. Every value is formed by the generic kernel's operations in its
// order (its blocks of ``per`` rows, its trees), so the basis, and with it
// every later rounding of a solve, is the same to the last bit.
constexpr int kNR16 = 16, kRows16 = 128;

// blockIdx.x = (virtual block, column group); warp w: rows 32 (w % 4) .., column w / 4 of the group
template <int CPB>
__global__ void __launch_bounds__(kRows16* CPB, 2) pcg16_kernel(PcgArgsT<double> a, int per, int nvb) {
  constexpr int kGroups = kNR16 / CPB;
  __shared__ double sVal[kEll][kRows16];
  __shared__ int32_t sCol[kEll][kRows16];
  __shared__ double s_red[4 * CPB][4];
  __shared__ double s_grp[4][4 * CPB];
  __shared__ double s_al[CPB], s_be[CPB];
  __shared__ int s_act[CPB], s_zero[CPB];
  __shared__ int s_flag, s_any;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int rw = warp & 3, jc = warp >> 2;
  const int vb = blockIdx.x / kGroups, cg = blockIdx.x % kGroups, j = cg * CPB + jc;
  const int64_t n = a.n;
  const int64_t r0 = (int64_t)vb * per, r1 = r0 + per < n ? r0 + per : n;
  const int nwr = r1 > r0 ? (int)((r1 - r0 + 31) / 32) : 0;
  const int lr = rw * 32 + lane;
  const bool own = r0 + lr < r1;
  const int64_t v = own ? r0 + lr : 0;
  double* __restrict__ ug = a.u + (size_t)j * n;
  double* __restrict__ part = a.partials;  // [virtual block][item][column]
  int* act = reinterpret_cast<int*>(part + (size_t)nvb * 64);  // per column group: still active
  unsigned epoch = 0;
  int cnt = 0;
  int32_t e0 = 0, e1 = 0;
  if (own) {
    e0 = __ldg(a.rowptr + v);
    e1 = __ldg(a.rowptr + v + 1);
    cnt = e1 - e0;
  }
  for (int t = jc; t < kEll; t += CPB) {
    sVal[t][lr] = t < cnt ? __ldg(a.val + e0 + t) : 0.0;
    sCol[t][lr] = t < cnt ? __ldg(a.col + e0 + t) : 0;
  }
  const double di = own ? __ldg(a.dinv + v) : 0.0;
  const double bv = own ? a.b[v * kNR16 + j] : 0.0;
  double x = own ? a.x[v * kNR16 + j] : 0.0;
  __syncthreads();
  auto spmv = [&](const double* z, int64_t stride) -> double {  // entries in the row's order, one accumulator
    double zz[kEll], acc = 0.0;
#pragma unroll
    for (int t = 0; t < kEll; ++t) zz[t] = t < cnt ? __ldcg(z + sCol[t][lr] * stride) : 0.0;
#pragma unroll
    for (int t = 0; t < kEll; ++t)
      if (t < cnt) acc = fma(sVal[t][lr], zz[t], acc);
    for (int32_t e = e0 + kEll; e < e1; ++e) acc = fma(__ldg(a.val + e), __ldcg(z + __ldg(a.col + e) * stride), acc);
    return acc;
  };
  // block sums of four items of this column into the virtual block's partials
  auto reduce = [&](double d0, double d1, double d2, double d3) {
    double t4[4] = {d0, d1, d2, d3};
    if (rw < nwr) {
      warp_halve<4>(t4, lane);
      if ((lane & 7) == 0) s_red[warp][lane >> 3] = t4[0];
    }
    __syncthreads();
    if (tid < 4 * CPB) {
      const int item = tid / CPB, c = tid % CPB;
      double t = 0.0;
      for (int g = 0; g < nwr; ++g) t += s_red[c * 4 + g][item];
      __stcg(part + (size_t)vb * 64 + item * kNR16 + cg * CPB + c, t);
    }
  };
  // sums over the virtual blocks: four groups take every fourth, then the
  // groups in order; thread item * CPB + c returns item ``item`` of column c
  auto gather_sums = [&]() -> double {
    if (tid < 16 * CPB) {
      const int k = tid % (4 * CPB), g = tid / (4 * CPB);
      const double* src = part + (k / CPB) * kNR16 + cg * CPB + k % CPB;
      double t = 0.0;
      for (int b = g; b < nvb; b += 32) {
        double l[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) l[q] = b + 4 * q < nvb ? __ldcg(src + (size_t)(b + 4 * q) * 64) : 0.0;
#pragma unroll
        for (int q = 0; q < 8; ++q)
          if (b + 4 * q < nvb) t += l[q];
      }
      s_grp[g][k] = t;
    }
    __syncthreads();
    double t = 0.0;
    if (tid < 4 * CPB)
      for (int g = 0; g < 4; ++g) t += s_grp[g][tid];
    __syncthreads();
    return t;
  };

  double r = own ? bv - spmv(a.x + j, kNR16) : 0.0;
  double u = di * r;
  if (own) __stcg(ug + v, u);
  if (!vbar(a.bar, epoch, &s_flag, a.wait_ns)) goto timeout;
  {
    double w = spmv(ug, 1);
    reduce(r * u, w * u, r * r, bv * bv);
    if (!vbar(a.bar, epoch, &s_flag, a.wait_ns)) goto timeout;
    // the scalars of column c in thread c, from the sums of threads c, CPB + c, ..
    double sga = 0.0, sal = 0.0, sthr = 0.0, sbb = 0.0, srr = 0.0;
    int sact = 0;
    double t = gather_sums();
    {
      const double dl = __shfl_sync(0xffffffffu, t, (lane + CPB) & 31), rr = __shfl_sync(0xffffffffu, t, (lane + 2 * CPB) & 31),
                   bb = __shfl_sync(0xffffffffu, t, (lane + 3 * CPB) & 31);
      if (tid < CPB) {
        sbb = bb;
        srr = rr;
        sthr = a.tol * a.tol * bb;
        sga = t;
        sact = (rr <= sthr || !(dl > 0.0)) ? 0 : 1;
        sal = sact ? t / dl : 0.0;
        s_al[tid] = sal;
        s_act[tid] = sact;
        s_zero[tid] = bb == 0.0;
      }
    }
    __syncthreads();
    double p = u, s = w;
    if (s_zero[jc]) x = 0.0;  // zero right-hand side: x = 0 exactly
    int it = 0;
    bool all_done = false;
    for (;;) {
      if (vb == 0 && tid == 0) {
        int on = 0;
        for (int c = 0; c < CPB; ++c) on |= s_act[c];
        __stcg(act + cg, on);
      }
      if (s_act[jc] && it < a.max_iter) {
        x = fma(s_al[jc], p, x);
        r = fma(-s_al[jc], s, r);
        u = di * r;
      }
      if (own) __stcg(ug + v, u);
      if (!vbar(a.bar, epoch, &s_flag, a.wait_ns)) goto timeout;
      // every block sees every group's state, so all leave together
      if (tid == 0) {
        int on = 0;
        for (int g = 0; g < kGroups; ++g) on |= __ldcg(act + g);
        s_any = on;
      }
      __syncthreads();
      all_done = s_any == 0;
      if (all_done || it >= a.max_iter) break;
      ++it;
      w = spmv(ug, 1);
      reduce(r * u, w * u, r * r, 0.0);
      if (!vbar(a.bar, epoch, &s_flag, a.wait_ns)) goto timeout;
      t = gather_sums();
      {
        const double dl = __shfl_sync(0xffffffffu, t, (lane + CPB) & 31), rr = __shfl_sync(0xffffffffu, t, (lane + 2 * CPB) & 31);
        if (tid < CPB && sact) {
          srr = rr;
          if (rr <= sthr) {
            sact = 0;
          } else {
            const double be = t / sga;
            const double den = dl - be * t / sal;
            if (!(den > 0.0)) {  // breakdown: stop this column
              sact = 0;
            } else {
              s_be[tid] = be;
              sal = t / den;
              s_al[tid] = sal;
              sga = t;
            }
          }
          s_act[tid] = sact;
        }
      }
      __syncthreads();
      if (s_act[jc]) {
        p = fma(s_be[jc], p, u);
        s = fma(s_be[jc], s, w);
      }
      __syncthreads();
    }
    if (own) a.x[v * kNR16 + j] = x;
    if (vb == 0 && tid < CPB && a.relres_out) a.relres_out[cg * CPB + tid] = sbb > 0.0 ? sqrt(srr / sbb) : 0.0;
    if (blockIdx.x == 0 && tid == 0) {
      if (a.iters_out) atomicAdd(a.iters_out, it);
      if (a.fail_out && !all_done) atomicExch(a.fail_out, 1);
      if (a.last_iters) *a.last_iters = it;
    }
  }
  vbar_exit(a.bar);
  return;
timeout:
  if (tid == 0 && a.timeout_out) atomicExch(a.timeout_out, 1);
  vbar_exit(a.bar);
}

namespace {
template <int CPB> cudaError_t launch16(const PcgArgsT<double>& args, int per, int nvb, cudaStream_t st) {
  PcgArgsT<double> a = args;
  void* params[] = {(void*)&a, (void*)&per, (void*)&nvb};
  return cudaLaunchCooperativeKernel((const void*)pcg16_kernel<CPB>, dim3(nvb * (kNR16 / CPB)), dim3(kRows16 * CPB),
                                     params, 0, st);
}
}  // namespace

// Columns per block so that the grid is about two blocks per SM; 0 where the
// 16 n threads of the kernel exceed 1,024 per SM, or the generic kernel's
// blocks (``grid`` of them) would hold more than 128 rows.
int pcg16_columns(int64_t n, int grid, int sms) {
  if (grid < 1 || n < 1 || kNR16 * n > 1024 * (int64_t)sms || (n + grid - 1) / grid > kRows16) return 0;
  for (int c = 1; c <= 4; c *= 2)
    if ((int64_t)grid * (kNR16 / c) <= 2 * (int64_t)sms) return c;
  return 0;
}

cudaError_t launch_pcg16(const PcgArgsT<double>& args, int grid, int columns, cudaStream_t st) {
  if (!args.bar_clean) {
    const cudaError_t e = cudaMemsetAsync(args.bar, 0, sizeof(GridBarrier), st);
    if (e != cudaSuccess) return e;
  }
  const int per = (int)((args.n + grid - 1) / grid);
  switch (columns) {
    case 1: return launch16<1>(args, per, grid, st);
    case 2: return launch16<2>(args, per, grid, st);
    default: return launch16<4>(args, per, grid, st);
  }
}

// Rows per block: the smallest multiple of 32 that needs at most one block
// per SM; false above 320 (n > 320 per SM: the generic kernel).
bool pcg64_shape(int64_t n, int sms, int* grid, int* rows) {
  if (sms < 1 || n < 1) return false;
  const int64_t r = std::max<int64_t>(1, (n + 32 * (int64_t)sms - 1) / (32 * (int64_t)sms)) * 32;
  if (r > kMaxRows) return false;
  *rows = (int)r;
  *grid = (int)((n + r - 1) / r);
  return true;
}

cudaError_t launch_pcg64(const PcgArgsT<double>& args, int grid, int rows, cudaStream_t st) {
  if (!args.bar_clean) {
    const cudaError_t e = cudaMemsetAsync(args.bar, 0, sizeof(GridBarrier), st);
    if (e != cudaSuccess) return e;
  }
  return args.phit ? pick64<true>(args, rows, grid, st) : pick64<false>(args, rows, grid, st);
}

// out[k n + v] = sum_l phi[v][l] T[l][k]: the coarse basis with T T^T = E^-1, mode-major
__global__ void __launch_bounds__(256) k_phit(int64_t n, const double* __restrict__ phi, const double* __restrict__ T,
                                              double* __restrict__ out) {
  __shared__ double sT[kModes * kModes];
  for (int e = threadIdx.x; e < kModes * kModes; e += blockDim.x) sT[e] = T[e];
  __syncthreads();
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n * kModes; i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t k = i / n, v = i % n;
    double acc = 0.0;
    for (int l = 0; l < kModes; ++l) acc = fma(phi[v * kModes + l], sT[l * kModes + k], acc);
    out[i] = acc;
  }
}

cudaError_t launch_phit(int64_t n, const double* phi, const double* T, double* out, cudaStream_t st) {
  const int grid = (int)std::min<int64_t>(std::max<int64_t>(1, (n * kModes + 255) / 256), 4096);
  k_phit<<<grid, 256, 0, st>>>(n, phi, T, out);
  return cudaGetLastError();
}

}  // namespace emu
