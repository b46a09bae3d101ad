// Per-tet and per-vertex kernels of one Newton iteration of EMU's
// quasi-static solve in rotation/stretch form (arXiv 2006.08821, Sec. 3).
//
// One iteration (the host drives the order, everything stays on the device):
//   rhs_from_state -> assemble -> PCG          q = q*(R S)              (Eq. 4)
//   grad            g = V P(F) + alpha w (F - G q), |g|^2, Uw, y = H^-1 g  (Eqs. 6-7)
//   syrk + cap      C = sum w (G Phi)^T N (G Phi), B y, z = C^-1 B y    (Eqs. 9-12)
//   dir             d = -(y + (I - N) (G Phi) z), corner RHS of G^T W d
//   assemble -> PCG dq = q*(d) linear part
//   ls + select     Armijo backtracking on E(F + sigma d)              (Algorithm 1)
//   update          F <- F + sigma d, polar re-extraction of R, S; q += sigma dq
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "emu_capslots.h"
#include "emu_kernels.cuh"
#include "emu_math.cuh"
#include "emu_reduce.cuh"
#include "emu_tetio.cuh"

namespace emu {

// ------------------------------------------------- coupling-solve RHS ----
__global__ void __launch_bounds__(256) k_rhs_from_state(TetArgs<double> a) {
  const int64_t m = a.m;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < m; i += (int64_t)gridDim.x * blockDim.x) {
    double D[9], R[9], sv[6], S[9], F[9];
    load_dinv(a.Dinv, m, i, D);
#pragma unroll
    for (int k = 0; k < 9; ++k) R[k] = a.R[k * m + i];
#pragma unroll
    for (int k = 0; k < 6; ++k) sv[k] = a.s[k * m + i];
    sym_from_s(sv, S);
    matmul3(R, S, F);
    write_corners(a.contrib, i, a.w[i], F, D);
  }
}

void launch_rhs_from_state(const TetArgs<double>& a, int grid, cudaStream_t st) {
  k_rhs_from_state<<<grid, 256, 0, st>>>(a);
}

// One thread per vertex and coordinate: the corner terms are added in slot
// order, eight in flight with the next eight indices, so a vertex of 24 corners
// costs four L2 round trips instead of a chain through every slot (425
// vertices 12.6 us, 1,485 in FP32 8.1 us before).
__global__ void __launch_bounds__(128) k_assemble(int64_t n, const int32_t* __restrict__ slot_ptr,
                                                  const int32_t* __restrict__ slot_idx,
                                                  const double* __restrict__ contrib, const double* __restrict__ bfix,
                                                  const uint8_t* __restrict__ is_fixed,
                                                  const double* __restrict__ qfix, int mode, double* __restrict__ b) {
  dep_sync();
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < 3 * n; i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t v = i / 3;
    double s = 0.0;
    if (is_fixed[v]) {
      if (mode == 0) s = qfix[i];
    } else {
      s = gather_corners(slot_idx, slot_ptr[v], slot_ptr[v + 1], contrib + (i - 3 * v));
      if (mode == 0) s -= bfix[i];
    }
    b[i] = s;
  }
}

void launch_assemble(int64_t n, const int32_t* slot_ptr, const int32_t* slot_idx, const double* contrib,
                     const double* bfix, const uint8_t* is_fixed, const double* qfix, int mode, double* b,
                     cudaStream_t st) {
  const int64_t grid = (3 * n + 127) / 128;
  launch_dep(n <= kDepTets / 2, k_assemble, (int)(grid < 1 ? 1 : grid), 128, 0, st, n, slot_ptr, slot_idx, contrib, bfix, is_fixed, qfix, mode, b);
}

// ------------------------------------------------------------ gradient ----
// g = V R Pr(S) + alpha w (R S - G_i q) in FP64 (Eqs. 6-7); the chart factor
// Uw and y = H_F^-1 g = (g - N g) / (alpha w) in TW.
template <typename TW>
__global__ void __launch_bounds__(128) k_grad(TetArgs<TW> a) {
  dep_sync();
  const int64_t m = a.m;
  double acc[1] = {0.0};
  int bad = 0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < m; i += (int64_t)gridDim.x * blockDim.x) {
    // tets of bones are no variables of their own (their g, y, U stay zero)
    if (a.tkind && a.tkind[i] != kTetDeformable) continue;
    const int4 t = a.tet[i];
    double D[9], R[9], sv[6], S[9], F[9], A[9];
    load_dinv(a.Dinv, m, i, D);
#pragma unroll
    for (int k = 0; k < 9; ++k) R[k] = a.R[k * m + i];
#pragma unroll
    for (int k = 0; k < 6; ++k) sv[k] = a.s[k * m + i];
    sym_from_s(sv, S);
    matmul3(R, S, F);
    gather_defgrad(a.q, t, D, A);
    const ElemMat<double> md = load_mat<double>(a.V, a.mu, a.lam, a.ka, a.u, m, i);
    const double c = a.c[i];
    double Pr[9], Sinv[9], lnJ;
    piola_rotated(S, md, Pr, Sinv, lnJ);
    double RP[9];
    matmul3(R, Pr, RP);
    double g[9];
    double gg = 0.0;
#pragma unroll
    for (int k = 0; k < 9; ++k) {
      g[k] = md.V * RP[k] + c * (F[k] - A[k]);
      if (a.nu) g[k] -= a.nu[k * m + i];  // external force (Sec. 3.4)
      gg += g[k] * g[k];
      a.g[k * m + i] = g[k];
    }
    if (!isfinite(gg)) bad = 1;
    acc[0] += gg;

    // Hessian / Woodbury quantities in TW
    TW Sw[9], Siw[9], Rw[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) {
      Sw[k] = (TW)S[k];
      Siw[k] = (TW)Sinv[k];
      Rw[k] = (TW)R[k];
    }
    const ElemMat<TW> mw = load_mat<TW>(a.V, a.mu, a.lam, a.ka, a.u, m, i);
    TW M6[36];
    stretch_hessian(Siw, (TW)lnJ, mw, M6);
    TW U[54];
    bool ok = true;
    chart_factor(Rw, Sw, M6, (TW)c, U, ok);
    if (!ok) bad = 1;
    TW yv[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) yv[k] = (TW)g[k];
    apply_I_minus_N(U, yv);
    const TW ic = (TW)inv_n(c);
#pragma unroll
    for (int k = 0; k < 9; ++k) a.y[k * m + i] = yv[k] * ic;
#pragma unroll
    for (int k = 0; k < 54; ++k) a.Uw[k * m + i] = U[k];
  }
  block_reduce_write<1>(acc, a.partials + blockIdx.x);
  if (bad) atomicExch(&a.sc->nonfinite, 1);
  grad_finish(a.sc, a.partials);
}

template <typename TW> void launch_grad(const TetArgs<TW>& a, int grid, int threads, cudaStream_t st) {
  launch_dep(a.m <= kDepTets, k_grad<TW>, grid, threads, 0, st, a);
}

// ------------------------------------------------------------ capacitance --
// C = sum_i w_i (G_i Phi^T)^T N_i (G_i Phi^T) = sum_i Yh_i^T Yh_i with
// Yh_i = sqrt(w_i) Uw_i (G_i Phi^T) (6 x 48): column 16 r + j of (G_i Phi^T) is
// the matrix e_r gam_j^T, so Yh[k][16r+j] = sqrt(w) sum_b Uw[k][3r+b] gam_j[b].
// Also B y = sum_i w_i (G_i Phi^T)^T y_i: By[16r+j] = sum_i w_i sum_b y[r][b] gam_j[b].
template <typename TW>
__global__ void __launch_bounds__(256) k_syrk(TetArgs<TW> a, double* __restrict__ cpart) {
  dep_sync();
  // tets per chunk: few in FP64, whose pipe takes 10 us per 8 tets, so that
  // the chunks of a small mesh spread evenly over the SMs (6,080 tets at two
  // blocks per SM: 10 chunks of 4 on every SM, before 48 or 24 tets)
  constexpr int CH = sizeof(TW) == 8 ? kSyrk64Chunk : 16;
  constexpr int KR = CH * 6;
  __shared__ TW sY[KR][kK + 1];
  __shared__ TW sU[CH][54];
  __shared__ TW sg[CH][48];
  __shared__ TW sy[CH][9];
  __shared__ double sw[CH];
  __shared__ TW ssw[CH];  // sqrt(w), once per tet
  const int tid = threadIdx.x;
  int tr = 0, tc = 0;
  const bool tile = lower_tile(tid, tr, tc);  // 5 of the 8 warps issue the product
  TW acc[3][3];  // per-block partial sums in TW; across blocks in FP64
#pragma unroll
  for (int p = 0; p < 3; ++p)
#pragma unroll
    for (int q = 0; q < 3; ++q) acc[p][q] = TW(0);
  double by = 0.0;
  const int64_t m = a.m;
  const int64_t nch = (m + CH - 1) / CH;
  for (int64_t ch = blockIdx.x; ch < nch; ch += gridDim.x) {
    const int64_t base = ch * CH;
    for (int e = tid; e < CH * 54; e += 256) {
      const int tt = e / 54, k = e % 54;
      const int64_t i = base + tt;
      sU[tt][k] = i < m ? a.Uw[k * m + i] : TW(0);
    }
    for (int e = tid; e < CH * 48; e += 256) {
      const int tt = e / 48, k = e % 48;
      const int64_t i = base + tt;
      sg[tt][k] = i < m ? a.gam[k * m + i] : TW(0);
    }
    for (int e = tid; e < CH * 9; e += 256) {
      const int tt = e / 9, k = e % 9;
      const int64_t i = base + tt;
      sy[tt][k] = i < m ? a.y[k * m + i] : TW(0);
    }
    if (tid < CH) {
      sw[tid] = (base + tid) < m ? a.w[base + tid] : 0.0;
      ssw[tid] = (TW)sqrt(sw[tid]);
    }
    __syncthreads();
    for (int e = tid; e < CH * 6 * kK; e += 256) {
      const int tt = e / (6 * kK), rem = e % (6 * kK);
      const int k = rem / kK, col = rem % kK;
      const int r = col >> 4, j = col & 15;
      TW v = sU[tt][9 * k + 3 * r] * sg[tt][3 * j] + sU[tt][9 * k + 3 * r + 1] * sg[tt][3 * j + 1] +
             sU[tt][9 * k + 3 * r + 2] * sg[tt][3 * j + 2];
      sY[tt * 6 + k][col] = v * ssw[tt];
    }
    __syncthreads();
#pragma unroll 4
    for (int kr = 0; kr < (tile ? KR : 0); ++kr) {
      const TW a0 = sY[kr][3 * tr], a1 = sY[kr][3 * tr + 1], a2 = sY[kr][3 * tr + 2];
      const TW b0 = sY[kr][3 * tc], b1 = sY[kr][3 * tc + 1], b2 = sY[kr][3 * tc + 2];
      acc[0][0] += a0 * b0;
      acc[0][1] += a0 * b1;
      acc[0][2] += a0 * b2;
      acc[1][0] += a1 * b0;
      acc[1][1] += a1 * b1;
      acc[1][2] += a1 * b2;
      acc[2][0] += a2 * b0;
      acc[2][1] += a2 * b1;
      acc[2][2] += a2 * b2;
    }
    if (tid < kK) {
      const int r = tid >> 4, j = tid & 15;
      for (int tt = 0; tt < CH; ++tt) {
        by += sw[tt] * ((double)sy[tt][3 * r] * (double)sg[tt][3 * j] + (double)sy[tt][3 * r + 1] * (double)sg[tt][3 * j + 1] +
                        (double)sy[tt][3 * r + 2] * (double)sg[tt][3 * j + 2]);
      }
    }
    __syncthreads();
  }
  // entry-major partials: cpart[e * gridDim.x + block]
  const size_t nb = gridDim.x;
  if (tile)
#pragma unroll
    for (int p = 0; p < 3; ++p)
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        const double v = (double)acc[p][q];
        cpart[(size_t)((3 * tr + p) * kK + 3 * tc + q) * nb + blockIdx.x] = v;
        if (tr != tc) cpart[(size_t)((3 * tc + q) * kK + 3 * tr + p) * nb + blockIdx.x] = v;
      }
  if (tid < kK) cpart[(size_t)(kCapEntries + tid) * nb + blockIdx.x] = by;
}

template <typename TW> void launch_syrk(const TetArgs<TW>& a, int grid, double* cpart, cudaStream_t st) {
  launch_dep(a.m <= kDepTets, k_syrk<TW>, grid, 256, 0, st, a, cpart);
}

// ------------------------------------------- capacitance sum and solve ----
__device__ __forceinline__ float pivot_inverse(float d) { return __frcp_rn(d); }
__device__ __forceinline__ double pivot_inverse(double d) { return inv_n(d); }

static_assert(kCapN == kK, "emu_capslots.h");
constexpr int kCapNB = 4;  // columns of a panel

// Sums the per-block partials of C (lower triangle) and B y, one warp per
// entry (entry-major, coalesced, a fixed shuffle tree), and in the last block
// to finish factors C = L D L^T and solves z = C^-1 (B y) in T arithmetic
// (FP64; FP32 for the mixed path, whose C comes from TF32 products).
//
// Latency decides here: one block, 48 dependent pivots. Each of the 256
// threads owns up to five entries of the lower triangle in registers, with
// B y as row 48, so the forward substitution is part of the factorisation.
// Per panel of four columns the owners hand the panel to two warps, which
// factor it with their rows in registers (shuffles instead of barriers), and
// every thread then applies the four rank-1 updates to its entries: two block
// barriers per four columns, and the work of the trailing triangle only. The
// entries are numbered from the last column backwards, so the trailing
// entries are a prefix and whole warps drop out as it shrinks. In FP64 a warp
// instruction holds an SM's FP64 pipe for 19 cycles: 1.1e4 cycles for the
// updates, and the pivots' reciprocals are Newton steps in one warp.
// Measured per Newton iteration with the reduction (event pairs around the
// phase, which add about 4 us to a launch): FP32 27 us as two launches with a
// barrier and a division per column, 20 to 22 us now; FP64 83 us, 34 us now.
template <typename T>
__global__ void __launch_bounds__(256) k_cap(const double* __restrict__ cpart, int nblk, double* __restrict__ cfull,
                                             const double* __restrict__ cadd, double* z, DevScalars* sc) {
  dep_sync();
  const int tid = threadIdx.x, lane = tid & 31;
  {
    const int e = blockIdx.x * 8 + (tid >> 5);
    if (e < kCapSums) {
      int src = kCapEntries + (e - kCapLow);  // of cpart: row-major 48 x 48, then B y
      if (e < kCapLow) {
        int i = (int)((sqrtf(8.f * e + 1.f) - 1.f) * 0.5f);
        while ((i + 1) * (i + 2) / 2 <= e) ++i;
        while (i * (i + 1) / 2 > e) --i;
        src = i * kK + (e - i * (i + 1) / 2);
      }
      double x = 0.0;
      for (int b = lane; b < nblk; b += 32) x += cpart[(size_t)src * nblk + b];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
      if (lane == 0) __stcg(cfull + src, cadd ? x + cadd[src] : x);
    }
  }
  int row[kCapOwn], col[kCapOwn];
#pragma unroll
  for (int s = 0; s < kCapOwn; ++s) cap_slot(tid, s, &row[s], &col[s]);
  if (!last_block(&sc->ticket[kTicketCap])) return;
  // In FP64 B y is row 48 of the factorisation, which leaves D^-1 L^-1 (B y)
  // there. In FP32 the third warp substitutes with 1 / sqrt(d) scaling while
  // the others update (the mixed path's rounding, and so its iterates, are
  // those of a plain column-by-column factorisation).
  constexpr bool kRowB = sizeof(T) == 8;
  __shared__ T sL[kK + 1][kK + 1];      // finished columns, scaled by 1 / d (FP32: unscaled)
  __shared__ T sP[kCapNB][kK + 1];      // the panel's columns
  __shared__ T sW[2][kCapNB][kK + 1];   // the finished columns of this and the last panel, unscaled
  __shared__ T sS[kCapNB][kK + 1];      // and scaled by 1 / d
  __shared__ T sR[kK];                  // FP32: 1 / sqrt(d)
  __shared__ int s_ok;
  T val[kCapOwn];
#pragma unroll
  for (int s = 0; s < kCapOwn; ++s) {
    const int c = col[s], src = cap_source(row[s], c);
    val[s] = T(0);
    if (src < 0) continue;  // a slot past the last entry
    val[s] = (T)__ldcg(cfull + src);
    // unused modes (k_modes < 48) have zero rows: identity rows with a zero right-hand side
    if (__ldcg(cfull + c * kK + c) == 0.0) val[s] = row[s] == c ? T(1) : row[s] == kK ? T(0) : val[s];
  }
  if (tid == 0) s_ok = 1;
  T x0 = T(0), x1 = T(0);  // FP32: right-hand side rows lane and 32 + lane of the third warp
  const bool has1 = lane + 32 < kK;
  if (!kRowB && tid >= 64 && tid < 96) {
    if (__ldcg(cfull + lane * kK + lane) != 0.0) x0 = (T)__ldcg(cfull + kCapEntries + lane);
    if (has1 && __ldcg(cfull + (lane + 32) * kK + lane + 32) != 0.0) x1 = (T)__ldcg(cfull + kCapEntries + lane + 32);
  }
  // L y = b, y_j = x_j / L_jj with L_ij = C_ij / sqrt(d_j) (FP32, the third
  // warp), for the columns of the panel at p0; the four roots in four lanes
  auto substitute = [&](int p0, const T (*W)[kK + 1]) {
    const T d4 = W[lane & (kCapNB - 1)][p0 + (lane & (kCapNB - 1))];
    const T ri4 = positive_n(d4) ? T(1) / sqrt(d4) : T(1);
    if (lane < kCapNB) sR[p0 + lane] = ri4;
#pragma unroll
    for (int p = 0; p < kCapNB; ++p) {
      const int j = p0 + p;
      const T ri = __shfl_sync(0xffffffffu, ri4, p);
      const T yj = __shfl_sync(0xffffffffu, j < 32 ? x0 : x1, j & 31) * ri;
      const T f = ri * yj;
      if (lane == (j & 31)) {
        if (j < 32) x0 = yj; else x1 = yj;
      }
      if (lane > j) x0 -= W[p][lane] * f;
      if (has1 && lane + 32 > j) x1 -= W[p][lane + 32] * f;
    }
  };
  for (int p0 = 0, buf = 0; p0 < kK; p0 += kCapNB, buf ^= 1) {
#pragma unroll
    for (int s = 0; s < kCapOwn; ++s)
      if (col[s] >= p0 && col[s] < p0 + kCapNB) sP[col[s] - p0][row[s]] = val[s];
    __syncthreads();
    if (tid < 64) {
      // row of this lane: warp 0 takes p0 .. p0 + 31; warp 1 copies of the
      // four pivot rows in its first lanes, then p0 + 32 ..
      const bool copy = tid >= 32 && lane < kCapNB;
      const int r = tid < 32 || copy ? p0 + lane : p0 + 32 - kCapNB + lane;
      const bool on = r <= kK && !copy;
      T v[kCapNB];
#pragma unroll
      for (int q = 0; q < kCapNB; ++q) v[q] = r <= kK && r >= p0 + q ? sP[q][r] : T(0);
#pragma unroll
      for (int p = 0; p < kCapNB; ++p) {
        T d = __shfl_sync(0xffffffffu, v[p], p);
        if (!positive_n(d)) {  // not positive definite: recorded, z = 0 below
          d = T(1);
          s_ok = 0;
        }
        const T l = v[p] * pivot_inverse(d);
        if (on) {
          sW[buf][p][r] = v[p];
          sS[p][r] = l;
          sL[r][p0 + p] = kRowB ? l : v[p];
        }
#pragma unroll
        for (int q = p + 1; q < kCapNB; ++q) v[q] -= l * __shfl_sync(0xffffffffu, v[p], q);
      }
    } else if (!kRowB && tid < 96 && p0 > 0) {
      substitute(p0 - kCapNB, sW[buf ^ 1]);  // one panel behind, while this one is factored
    }
    __syncthreads();
#pragma unroll
    for (int s = 0; s < kCapOwn; ++s)
      if (col[s] >= p0 + kCapNB) {
#pragma unroll
        for (int q = 0; q < kCapNB; ++q) val[s] -= sS[q][row[s]] * sW[buf][q][col[s]];
      }
  }
  if (tid < 64 || tid >= 96) return;
  if constexpr (kRowB) {  // L^T z = y with L unit lower triangular
    x0 = sL[kK][lane];
    if (has1) x1 = sL[kK][lane + 32];
#pragma unroll 4
    for (int j = kK - 1; j >= 32; --j) {
      const T zj = __shfl_sync(0xffffffffu, x1, j & 31);
      x0 -= sL[j][lane] * zj;
      if (lane + 32 < j) x1 -= sL[j][lane + 32] * zj;
    }
#pragma unroll 4
    for (int j = 31; j > 0; --j) {
      const T zj = __shfl_sync(0xffffffffu, x0, j);
      if (lane < j) x0 -= sL[j][lane] * zj;
    }
  } else {  // z_j = x_j / L_jj, then x_i -= L_ji z_j for i < j
    substitute(kK - kCapNB, sW[(kK / kCapNB - 1) & 1]);
    __syncwarp();
    const T r0 = sR[lane], r1 = has1 ? sR[lane + 32] : T(0);
#pragma unroll 4
    for (int j = kK - 1; j >= 32; --j) {
      const T zj = __shfl_sync(0xffffffffu, x1, j & 31) * sR[j];
      if (lane == (j & 31)) x1 = zj;
      x0 -= sL[j][lane] * r0 * zj;
      if (lane + 32 < j) x1 -= sL[j][lane + 32] * r1 * zj;
    }
#pragma unroll 4
    for (int j = 31; j >= 0; --j) {
      const T zj = __shfl_sync(0xffffffffu, x0, j) * sR[j];
      if (lane == j) x0 = zj;
      if (lane < j) x0 -= sL[j][lane] * r0 * zj;
    }
  }
  const int ok = s_ok;
  z[lane] = ok ? (double)x0 : 0.0;
  if (has1) z[lane + 32] = ok ? (double)x1 : 0.0;
  if (lane == 0) {
    sc->cap_ok = ok ? 1.0 : 0.0;
    sc->ticket[kTicketCap] = 0u;
  }
}

__global__ void k_ls_reset(DevScalars* sc, double sigma0) {
  sc->ls_fail = 0;
  sc->sigma_start = sigma0;
}

void launch_ls_reset(DevScalars* sc, double sigma0, cudaStream_t st) { k_ls_reset<<<1, 1, 0, st>>>(sc, sigma0); }

void launch_cap_solve(const double* cpart, int nblk, const double* cfull_scratch, double* z, DevScalars* sc,
                      bool fp32_factor, cudaStream_t st, const double* cadd) {
  double* cfull = const_cast<double*>(cfull_scratch);
  const int grid = (kCapSums + 7) / 8;
  if (fp32_factor)
    launch_dep(nblk <= kDepTets / 32, k_cap<float>, grid, 256, 0, st, cpart, nblk, cfull, cadd, z, sc);
  else
    launch_dep(nblk <= kDepTets / 32, k_cap<double>, grid, 256, 0, st, cpart, nblk, cfull, cadd, z, sc);
}

// ------------------------------------------------------------ direction ---
// d = -(y + alpha H_F^-1 w (G Phi^T) z) = -(y + (I - N) v), v = (G_i Phi^T) z.
template <typename TW>
__global__ void __launch_bounds__(128) k_dir(TetArgs<TW> a) {
  dep_sync();
  __shared__ double sz[kK];
  for (int k = threadIdx.x; k < kK; k += blockDim.x) sz[k] = a.z[k];
  __syncthreads();
  const int64_t m = a.m;
  double acc[1] = {0.0};
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < m; i += (int64_t)gridDim.x * blockDim.x) {
    if (a.tkind) {
      const int32_t kind = a.tkind[i];
      if (kind != kTetDeformable) {
        // a free bone's tet takes the bone's direction, a pinned bone's tet
        // none; their g . d is the bone's (summed by the bone kernel)
        double dv[9], D[9];
#pragma unroll
        for (int k = 0; k < 9; ++k) {
          dv[k] = kind >= 0 ? a.bone_st[(size_t)kind * kBoneStride + kBoneD + k] : 0.0;
          a.d[k * m + i] = (TW)dv[k];
        }
        load_dinv(a.Dinv, m, i, D);
        write_corners(a.contrib, i, a.w[i], dv, D);
        continue;
      }
    }
    TW gm[48];
#pragma unroll
    for (int k = 0; k < 48; ++k) gm[k] = a.gam[k * m + i];
    TW v[9];
#pragma unroll
    for (int r = 0; r < 3; ++r)
#pragma unroll
      for (int cc = 0; cc < 3; ++cc) {
        TW x = TW(0);
#pragma unroll
        for (int j = 0; j < 16; ++j) x += (TW)sz[16 * r + j] * gm[3 * j + cc];
        v[3 * r + cc] = x;
      }
    TW U[54];
#pragma unroll
    for (int k = 0; k < 54; ++k) U[k] = a.Uw[k * m + i];
    apply_I_minus_N(U, v);
    TW dv[9];
    double gtd = 0.0;
#pragma unroll
    for (int k = 0; k < 9; ++k) {
      dv[k] = -(a.y[k * m + i] + v[k]);
      a.d[k * m + i] = dv[k];
      gtd += a.g[k * m + i] * (double)dv[k];
    }
    acc[0] += gtd;
    double D[9];
    load_dinv(a.Dinv, m, i, D);
    write_corners(a.contrib, i, a.w[i], dv, D);
  }
  block_reduce_write<1>(acc, a.partials + blockIdx.x);
}

template <typename TW> void launch_dir(const TetArgs<TW>& a, int grid, int threads, cudaStream_t st) {
  launch_dep(a.m <= kDepTets, k_dir<TW>, grid, threads, 0, st, a);
}

// ------------------------------------------------------------ line search --
// Per trial sigma_j = sigma_start rho^j: V [Psi(F + sigma d) - Psi(F)] in FP64,
// written term by term (Algorithm 1's Armijo test needs the difference
// itself): with M = F^-1 d, ln det(I + sigma M) = log1p(sigma tr M
// + sigma^2 e2(M) + sigma^3 det M). The ACAP part is the exact quadratic
// alpha/2 sum w |D + sigma dD|^2 - |D|^2, D = G q - F, dD = G dq - d.
template <typename TW>
__global__ void __launch_bounds__(128) k_ls(TetArgs<TW> a, LsSelect sel) {
  dep_sync();
  const double rho = sel.rho;
  const int64_t m = a.m;
  const double s0 = a.sc->sigma_start;
  double acc[kLsNV];
#pragma unroll
  for (int k = 0; k < kLsNV; ++k) acc[k] = 0.0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < m; i += (int64_t)gridDim.x * blockDim.x) {
    // free bones' tets: once per bone in the bone kernel; pinned bones' tets contribute 0
    if (a.tkind && a.tkind[i] != kTetDeformable) continue;
    const int4 t = a.tet[i];
    double D9[9], R[9], sv[6], S[9], F[9], A[9], dA[9], d[9];
    load_dinv(a.Dinv, m, i, D9);
#pragma unroll
    for (int k = 0; k < 9; ++k) R[k] = a.R[k * m + i];
#pragma unroll
    for (int k = 0; k < 6; ++k) sv[k] = a.s[k * m + i];
#pragma unroll
    for (int k = 0; k < 9; ++k) d[k] = (double)a.d[k * m + i];
    sym_from_s(sv, S);
    matmul3(R, S, F);
    gather_defgrad(a.q, t, D9, A);
    gather_defgrad(a.dq, t, D9, dA);
    const double c = a.c[i];
    double cDd = 0.0, cdd = 0.0;
#pragma unroll
    for (int k = 0; k < 9; ++k) {
      const double Dk = A[k] - F[k], dDk = dA[k] - d[k];
      cDd += Dk * dDk;
      cdd += dDk * dDk;
    }
    acc[kLsTrials] += c * cDd;
    acc[kLsTrials + 1] += c * cdd;
    const ElemMat<double> md = load_mat<double>(a.V, a.mu, a.lam, a.ka, a.u, m, i);
    double Sinv[9];
    const double J = inv3(S, Sinv);
    const double lnJ = log(J);
    double Rtd[9], M[9];
    matTmul3(R, d, Rtd);
    matmul3(Sinv, Rtd, M);
    const double trM = M[0] + M[4] + M[8];
    const double e2 = inv2(M);
    const double detM = det3(M);
    // <F - F^-T, d> = <S - S^-1, R^T d>: the O(|d|) parts of mu <F, d> and
    // mu tr(F^-1 d) cancel before they are formed (a stiff, barely strained
    // element, a bone, would otherwise keep only their rounding)
    double FFd = 0.0, dd = 0.0;
#pragma unroll
    for (int k = 0; k < 9; ++k) {
      FFd += (S[k] - Sinv[k]) * Rtd[k];
      dd += d[k] * d[k];
    }
    double Fu[3], du[3];
#pragma unroll
    for (int r = 0; r < 3; ++r) {
      Fu[r] = F[3 * r] * md.u[0] + F[3 * r + 1] * md.u[1] + F[3 * r + 2] * md.u[2];
      du[r] = d[3 * r] * md.u[0] + d[3 * r + 1] * md.u[1] + d[3 * r + 2] * md.u[2];
    }
    const double Fudu = Fu[0] * du[0] + Fu[1] * du[1] + Fu[2] * du[2];
    const double dudu = du[0] * du[0] + du[1] * du[1] + du[2] * du[2];
    double dnu = 0.0;  // <d, nu>: the external work's change is -sigma <d, nu>
    if (a.nu)
#pragma unroll
      for (int k = 0; k < 9; ++k) dnu += d[k] * a.nu[k * m + i];
    double sig = s0;
#pragma unroll
    for (int j = 0; j < kLsTrials; ++j) {
      const double x = sig * trM + sig * sig * e2 + sig * sig * sig * detM;
      double dpsi;
      if (x > -1.0) {
        // mu [s <F, d> + s^2 |d|^2 / 2 - log1p(x)] with log1p(x) = x - (x - log1p x)
        const double xml = x_minus_log1p(x), dl = log1p_from(x, xml);
        const double nh = sig * FFd + 0.5 * sig * sig * dd - sig * sig * e2 - sig * sig * sig * detM + xml;
        dpsi = md.mu * nh + 0.5 * md.lam * dl * (2.0 * lnJ + dl) + md.ka * (2.0 * sig * Fudu + sig * sig * dudu);
        dpsi = dpsi * md.V - sig * dnu;
      } else {
        dpsi = 1e300;
      }
      acc[j] += dpsi;
      sig *= rho;
    }
  }
  block_reduce_write<kLsNV>(acc, a.partials + (size_t)blockIdx.x * kLsNV);
  ls_finish(a.sc, a.partials, sel);
}

template <typename TW> void launch_ls(const TetArgs<TW>& a, int grid, int threads, const LsSelect& sel, cudaStream_t st) {
  launch_dep(a.m <= kDepTets, k_ls<TW>, grid, threads, 0, st, a, sel);
}

// ------------------------------------------------------------ update ------
// F' = R S + sigma d; X = R^T F' = S + sigma R^T d is nearly symmetric, so its
// polar factor Rx is close to I; R' = R Rx, S' = sym(Rx^T X).
template <typename TW>
__global__ void __launch_bounds__(128) k_update_tets(TetArgs<TW> a, double* __restrict__ q) {
  dep_sync();
  const double sig = a.sc->sigma;
  if (sig == 0.0) return;
  const int64_t m = a.m;
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < 3 * a.n; k += (int64_t)gridDim.x * blockDim.x)
    q[k] += sig * a.dq[k];
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < m; i += (int64_t)gridDim.x * blockDim.x) {
    double R[9], sv[6], S[9], d[9], Rtd[9], X[9], Rx[9], Rn[9], Sn[9], sn[6];
#pragma unroll
    for (int k = 0; k < 9; ++k) R[k] = a.R[k * m + i];
#pragma unroll
    for (int k = 0; k < 6; ++k) sv[k] = a.s[k * m + i];
#pragma unroll
    for (int k = 0; k < 9; ++k) d[k] = (double)a.d[k * m + i];
    sym_from_s(sv, S);
    matTmul3(R, d, Rtd);
#pragma unroll
    for (int k = 0; k < 9; ++k) X[k] = S[k] + sig * Rtd[k];
    polar_rotation(X, Rx, 1e-15, 40);
    matTmul3(Rx, X, Sn);
    s_from_mat(Sn, sn);
    matmul3(R, Rx, Rn);
#pragma unroll
    for (int k = 0; k < 9; ++k) a.R[k * m + i] = Rn[k];
#pragma unroll
    for (int k = 0; k < 6; ++k) a.s[k * m + i] = sn[k];
  }
}

template <typename TW> void launch_update_tets(const TetArgs<TW>& a, int grid, int threads, double* q, cudaStream_t st) {
  launch_dep(a.m <= kDepTets, k_update_tets<TW>, grid, threads, 0, st, a, q);
}

// ------------------------------------------------------------ normaliser --
// ||g(F = I, q0)||: g = V * 2 ka u u^T + alpha w (I - G q0) (the neo-Hookean
// stress vanishes at I).
__global__ void __launch_bounds__(128) k_gref(TetArgs<double> a, const double* q0, double* partials) {
  const int64_t m = a.m;
  double acc[1] = {0.0};
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < m; i += (int64_t)gridDim.x * blockDim.x) {
    if (a.tkind && a.tkind[i] != kTetDeformable) continue;  // bones: summed per bone elsewhere
    double D[9], A[9];
    load_dinv(a.Dinv, m, i, D);
    gather_defgrad(q0, a.tet[i], D, A);
    const double V = a.V[i], c = a.c[i], ka = a.ka[i];
    const double u[3] = {a.u[i], a.u[m + i], a.u[2 * m + i]};
    double gg = 0.0;
#pragma unroll
    for (int r = 0; r < 3; ++r)
#pragma unroll
      for (int cc = 0; cc < 3; ++cc) {
        double gv = V * 2.0 * ka * u[r] * u[cc] + c * ((r == cc ? 1.0 : 0.0) - A[3 * r + cc]);
        if (a.nu) gv -= a.nu[(3 * r + cc) * m + i];
        gg += gv * gv;
      }
    acc[0] += gg;
  }
  block_reduce_write<1>(acc, partials + blockIdx.x);
}

__global__ void __launch_bounds__(256) k_sum_scalar(const double* partials, int nblk, double* out) {
  __shared__ double tot[1];
  block_sum_partials<1>(partials, nblk, tot);
  if (threadIdx.x == 0) out[0] = tot[0];
}

void launch_gref(const TetArgs<double>& a, const double* q0, int grid, double* partials, double* out,
                 cudaStream_t st) {
  k_gref<<<grid, 128, 0, st>>>(a, q0, partials);
  k_sum_scalar<<<1, 256, 0, st>>>(partials, grid, out);
}

// ------------------------------------------------------------ modes -------
__global__ void __launch_bounds__(256) k_gram16(int64_t n, const double* __restrict__ X, double* partials) {
  const int a = threadIdx.x >> 4, b = threadIdx.x & 15;
  const int64_t per = (n + gridDim.x - 1) / gridDim.x;
  const int64_t v0 = blockIdx.x * per;
  const int64_t v1 = v0 + per < n ? v0 + per : n;
  double acc = 0.0;
  for (int64_t v = v0; v < v1; ++v) acc += X[v * 16 + a] * X[v * 16 + b];
  partials[(size_t)blockIdx.x * 256 + threadIdx.x] = acc;
}

void launch_gram16(int64_t n, const double* X, int grid, double* partials, cudaStream_t st) {
  k_gram16<<<grid, 256, 0, st>>>(n, X, partials);
}

// Y = L X for 16 columns (L in CSR, X and Y vertex-major n x 16)
__global__ void __launch_bounds__(256) k_spmv16(int64_t n, const int32_t* __restrict__ rowptr,
                                                const int32_t* __restrict__ col, const double* __restrict__ val,
                                                const double* __restrict__ X, double* __restrict__ Y) {
  for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x) {
    double acc[16];
#pragma unroll
    for (int j = 0; j < 16; ++j) acc[j] = 0.0;
    for (int32_t e = rowptr[v]; e < rowptr[v + 1]; ++e) {
      const double a = val[e];
      const int64_t c = col[e];
#pragma unroll
      for (int j = 0; j < 16; ++j) acc[j] += a * X[c * 16 + j];
    }
#pragma unroll
    for (int j = 0; j < 16; ++j) Y[v * 16 + j] = acc[j];
  }
}

// partials of X^T Y (16 x 16) over contiguous vertex ranges
__global__ void __launch_bounds__(256) k_cross16(int64_t n, const double* __restrict__ X, const double* __restrict__ Y,
                                                 double* partials) {
  const int a = threadIdx.x >> 4, b = threadIdx.x & 15;
  const int64_t per = (n + gridDim.x - 1) / gridDim.x;
  const int64_t v0 = blockIdx.x * per;
  const int64_t v1 = v0 + per < n ? v0 + per : n;
  double acc = 0.0;
  for (int64_t v = v0; v < v1; ++v) acc += X[v * 16 + a] * Y[v * 16 + b];
  partials[(size_t)blockIdx.x * 256 + threadIdx.x] = acc;
}

void launch_galerkin16(int64_t n, const int32_t* rowptr, const int32_t* col, const double* val, const double* X,
                       double* Y, int grid, double* partials, cudaStream_t st) {
  int g2 = (int)((n + 255) / 256);
  if (g2 < 1) g2 = 1;
  k_spmv16<<<g2, 256, 0, st>>>(n, rowptr, col, val, X, Y);
  k_cross16<<<grid, 256, 0, st>>>(n, X, Y, partials);
}

__global__ void k_d2f(int64_t k, const double* a, float* b) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < k; i += (int64_t)gridDim.x * blockDim.x)
    b[i] = (float)a[i];
}

void launch_d2f(int64_t k, const double* a, float* b, cudaStream_t st) {
  int grid = (int)((k + 255) / 256);
  if (grid < 1) grid = 1;
  k_d2f<<<grid, 256, 0, st>>>(k, a, b);
}

__global__ void k_reduce_cols(const double* partials, int nblk, int nv, double* out) {
  for (int k = threadIdx.x; k < nv; k += blockDim.x) {
    double x = 0.0;
    for (int b = 0; b < nblk; ++b) x += partials[(size_t)b * nv + k];
    out[k] = x;
  }
}

void launch_reduce_cols(const double* partials, int nblk, int nv, double* out, cudaStream_t st) {
  k_reduce_cols<<<1, 256, 0, st>>>(partials, nblk, nv, out);
}

__global__ void __launch_bounds__(256) k_xform16(int64_t n, const double* __restrict__ T, double* X) {
  __shared__ double sT[256];
  sT[threadIdx.x] = T[threadIdx.x];
  __syncthreads();
  for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x) {
    double x[16], y[16];
#pragma unroll
    for (int k = 0; k < 16; ++k) x[k] = X[v * 16 + k];
#pragma unroll
    for (int j = 0; j < 16; ++j) {
      double s = 0.0;
#pragma unroll
      for (int k = 0; k < 16; ++k) s += x[k] * sT[16 * k + j];
      y[j] = s;
    }
#pragma unroll
    for (int k = 0; k < 16; ++k) X[v * 16 + k] = y[k];
  }
}

void launch_xform16(int64_t n, const double* T, double* X, cudaStream_t st) {
  int grid = (int)((n + 255) / 256);
  if (grid < 1) grid = 1;
  k_xform16<<<grid, 256, 0, st>>>(n, T, X);
}

// gam_j = gradient of mode j on tet i: sum_k (phi_j(v_k) - phi_j(v_3)) Dinv[k][:]
template <typename TW>
__global__ void __launch_bounds__(256) k_gamma(int64_t m, const int4* __restrict__ tet, const double* __restrict__ Dinv,
                                               const double* __restrict__ X, TW* gam) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < m; i += (int64_t)gridDim.x * blockDim.x) {
    const int4 t = tet[i];
    double D[9];
    load_dinv(Dinv, m, i, D);
    for (int j = 0; j < 16; ++j) {
      const double x3 = X[(int64_t)t.w * 16 + j];
      const double e0 = X[(int64_t)t.x * 16 + j] - x3;
      const double e1 = X[(int64_t)t.y * 16 + j] - x3;
      const double e2 = X[(int64_t)t.z * 16 + j] - x3;
#pragma unroll
      for (int c = 0; c < 3; ++c) gam[(3 * j + c) * m + i] = (TW)(e0 * D[c] + e1 * D[3 + c] + e2 * D[6 + c]);
    }
  }
}

template <typename TW>
void launch_gamma(int64_t m, const int4* tet, const double* Dinv, const double* X, TW* gam, cudaStream_t st) {
  int grid = (int)((m + 255) / 256);
  if (grid < 1) grid = 1;
  k_gamma<TW><<<grid, 256, 0, st>>>(m, tet, Dinv, X, gam);
}

// ------------------------------------------------------- external force ---
__global__ void __launch_bounds__(256) k_nu(int64_t m, const int4* __restrict__ tet, const double* __restrict__ Dinv,
                                            const double* __restrict__ w, const double* __restrict__ x,
                                            double* __restrict__ nu64, float* __restrict__ nu32) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < m; i += (int64_t)gridDim.x * blockDim.x) {
    double D[9], A[9];
    load_dinv(Dinv, m, i, D);
    gather_defgrad(x, tet[i], D, A);
    const double wi = w[i];
#pragma unroll
    for (int k = 0; k < 9; ++k) {
      const double v = wi * A[k];
      nu64[k * m + i] = v;
      if (nu32) nu32[k * m + i] = (float)v;
    }
  }
}

void launch_nu(int64_t m, const int4* tet, const double* Dinv, const double* w, const double* x, double* nu64,
               float* nu32, cudaStream_t st) {
  int grid = (int)((m + 255) / 256);
  if (grid < 1) grid = 1;
  k_nu<<<grid, 256, 0, st>>>(m, tet, Dinv, w, x, nu64, nu32);
}

// ------------------------------------------------------------ element API --
template <typename T>
__global__ void k_eval_stretch(const double* s, const double* prm, int64_t n, double* psi, double* grad, double* hess) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    T sv[6], S[9], Sinv[9];
#pragma unroll
    for (int k = 0; k < 6; ++k) sv[k] = (T)s[6 * i + k];
    ElemMat<T> e;
    e.V = (T)prm[8 * i];
    e.mu = (T)prm[8 * i + 1];
    e.lam = (T)prm[8 * i + 2];
    e.ka = (T)prm[8 * i + 3];
    e.u[0] = (T)prm[8 * i + 4];
    e.u[1] = (T)prm[8 * i + 5];
    e.u[2] = (T)prm[8 * i + 6];
    sym_from_s(sv, S);
    const T J = inv3(S, Sinv);
    const T lnJ = log(J);
    if (psi) psi[i] = (double)(e.V * psi_stretch(S, e));
    if (grad) {
      T g[6];
      stretch_gradient(S, Sinv, lnJ, e, g);
#pragma unroll
      for (int k = 0; k < 6; ++k) grad[6 * i + k] = (double)g[k];
    }
    if (hess) {
      T H[36];
      stretch_hessian(Sinv, lnJ, e, H);
#pragma unroll
      for (int k = 0; k < 36; ++k) hess[36 * i + k] = (double)H[k];
    }
  }
}

void launch_eval_stretch(const double* s, const double* prm, int64_t n, int mixed, double* psi, double* grad,
                         double* hess, cudaStream_t st) {
  int grid = (int)((n + 127) / 128);
  if (grid < 1) grid = 1;
  if (mixed)
    k_eval_stretch<float><<<grid, 128, 0, st>>>(s, prm, n, psi, grad, hess);
  else
    k_eval_stretch<double><<<grid, 128, 0, st>>>(s, prm, n, psi, grad, hess);
}

__global__ void k_eval_polar(const double* F, int64_t n, double* R, double* s) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    double X[9], Rr[9], S[9], sv[6];
#pragma unroll
    for (int k = 0; k < 9; ++k) X[k] = F[9 * i + k];
    polar_rotation(X, Rr, 1e-15, 60);
    matTmul3(Rr, X, S);
    s_from_mat(S, sv);
#pragma unroll
    for (int k = 0; k < 9; ++k) R[9 * i + k] = Rr[k];
#pragma unroll
    for (int k = 0; k < 6; ++k) s[6 * i + k] = sv[k];
  }
}

void launch_eval_polar(const double* F, int64_t n, double* R, double* s, cudaStream_t st) {
  int grid = (int)((n + 127) / 128);
  if (grid < 1) grid = 1;
  k_eval_polar<<<grid, 128, 0, st>>>(F, n, R, s);
}

// F may alias R: each thread reads its tet's R before it writes F.
__global__ void k_compose_F(int64_t m, const double* R, const double* s, double* F) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < m; i += (int64_t)gridDim.x * blockDim.x) {
    double Rr[9], sv[6], S[9], Fi[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) Rr[k] = R[k * m + i];
#pragma unroll
    for (int k = 0; k < 6; ++k) sv[k] = s[k * m + i];
    sym_from_s(sv, S);
    matmul3(Rr, S, Fi);
#pragma unroll
    for (int k = 0; k < 9; ++k) F[k * m + i] = Fi[k];
  }
}

void launch_compose_F(int64_t m, const double* R, const double* s, double* F, cudaStream_t st) {
  int grid = (int)((m + 255) / 256);
  if (grid < 1) grid = 1;
  k_compose_F<<<grid, 256, 0, st>>>(m, R, s, F);
}

// explicit instantiations
template void launch_grad<double>(const TetArgs<double>&, int, int, cudaStream_t);
template void launch_syrk<double>(const TetArgs<double>&, int, double*, cudaStream_t);
template void launch_dir<double>(const TetArgs<double>&, int, int, cudaStream_t);
template void launch_ls<double>(const TetArgs<double>&, int, int, const LsSelect&, cudaStream_t);
template void launch_update_tets<double>(const TetArgs<double>&, int, int, double*, cudaStream_t);
template void launch_gamma<double>(int64_t, const int4*, const double*, const double*, double*, cudaStream_t);
template void launch_gamma<float>(int64_t, const int4*, const double*, const double*, float*, cudaStream_t);

}  // namespace emu
