// Building blocks of a Lanczos step run by a cooperative grid (CTA g owns the contiguous slice
// [e0, e0 + len) of every vector): a bounded grid barrier, per-slice dot products against the
// Krylov basis, fixed-order cross-CTA reductions that every CTA evaluates identically, the
// projection, the norm, and the tridiagonal bookkeeping with the small exponential.  Used by
// the fused bond exponential (bond_krylov.cu) and the fused site-Lanczos step
// (lanczos_step.cu).  All sums have a fixed order, so results do not depend on timing.
#pragma once

#include "fp64_util.cuh"
#include "lanczos_exp.cuh"
#include "tdmrg_internal.cuh"

namespace tdmrg {
namespace lzc {

constexpr int NV = KMAX + 1;                      // partial-dot slots per CTA

__device__ __forceinline__ double wsum(double v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Grid barrier on one monotonic counter: barrier number e is passed once the counter reaches
// e * nblocks (one atomic per CTA; the launcher clears the counter).  Bounded: gives up after
// `limit` clock cycles (kBarrierWaitCycles, ~2 s, unless a test lowers it), sets *status = 1,
// and every CTA then leaves.
__device__ __forceinline__ bool barrier(unsigned* bar, unsigned nblocks, unsigned& epoch,
                                        int* status, long long limit) {
  __syncthreads();
  __shared__ int s_ok;
  ++epoch;
  if (threadIdx.x == 0) {
    volatile unsigned* vbar = bar;
    volatile int* vstat = status;
    const unsigned target = epoch * nblocks;
    __threadfence();
    atomicAdd(bar, 1u);
    int ok = 1;
    const long long t0 = clock64();
    while (*vbar < target) {
      if (*vstat) { ok = 0; break; }
      if (clock64() - t0 > limit) {
        atomicExch(status, 1);
        ok = 0;
        break;
      }
    }
    __threadfence();
    s_ok = ok;
  }
  __syncthreads();
  return s_ok != 0;
}

// Warp wv computes the partial dots conj(q_i) . w over the own slice for i = i0 + wv,
// i0 + wv + nwarps, ... < i1 (lanes stride the slice, fixed warp tree) and stores them at
// part[blockIdx.x * NV + i].  V holds the basis (vector i at V + i * n); w points at the own
// slice of w (shared or global memory).
__device__ __forceinline__ void slice_dots(const cplx* V, long long n, const cplx* w,
                                           long long e0, int len, int i0, int i1, cplx* part) {
  const int lane = threadIdx.x & 31, wv = threadIdx.x >> 5, nw = blockDim.x >> 5;
  for (int i = i0 + wv; i < i1; i += nw) {
    const cplx* q = V + (size_t)i * n + e0;
    double sr = 0.0, si = 0.0;
    for (int e = lane; e < len; e += 32) {
      const cplx a = q[e], b = w[e];
      sr = fma(a.x, b.x, sr);
      sr = fma(a.y, b.y, sr);
      si = fma(a.x, b.y, si);
      si = fma(-a.y, b.x, si);
    }
    sr = wsum(sr);
    si = wsum(si);
    if (lane == 0) part[(size_t)blockIdx.x * NV + i] = make_double2(sr, si);
  }
}

// The same partial dots with every thread of the CTA on every vector (for large slices), and with
// `norm` the slice's ||w||^2: the vectors are taken four at a time, each thread sums its elements
// (stride blockDim), the threads of a warp are added by a tree (lane offsets 16 .. 1), the warps in
// order.  One warp forms the trees of one value for all warps, halving the values it holds at every
// offset: 16 FP64 additions of a warp where a tree in every warp takes 80, with the same bits (the
// order is part of the result: C(t) of a truncated chain on the mixed path follows the last bit).
// red: 9 * blockDim doubles of shared memory; blockDim is 512.
__device__ __forceinline__ void slice_dots_block(const cplx* V, long long n, const cplx* w,
                                                 long long e0, int len, int i0, int i1,
                                                 cplx* part, double* norm, double* red) {
  constexpr int T = 512, nw = T / 32;
  const int lane = threadIdx.x & 31, wv = threadIdx.x >> 5;
  for (int c0 = i0; c0 < i1; c0 += 4) {
    const int nv = min(4, i1 - c0);
    const bool nrm = norm && c0 == i0;
    double sr[4] = {0.0, 0.0, 0.0, 0.0}, si[4] = {0.0, 0.0, 0.0, 0.0}, sn = 0.0;
    for (int e = threadIdx.x; e < len; e += T) {
      const cplx b = w[e];
      if (nrm) sn = fma(b.x, b.x, fma(b.y, b.y, sn));
#pragma unroll
      for (int v = 0; v < 4; ++v) {
        if (v < nv) {
          const cplx a = V[(size_t)(c0 + v) * n + e0 + e];
          sr[v] = fma(a.x, b.x, sr[v]);
          sr[v] = fma(a.y, b.y, sr[v]);
          si[v] = fma(a.x, b.y, si[v]);
          si[v] = fma(-a.y, b.x, si[v]);
        }
      }
    }
#pragma unroll
    for (int v = 0; v < 4; ++v)
      if (v < nv) {
        red[(2 * v) * T + threadIdx.x] = sr[v];
        red[(2 * v + 1) * T + threadIdx.x] = si[v];
      }
    if (nrm) red[8 * T + threadIdx.x] = sn;
    __syncthreads();
    const int live = min(T, len);                   // threads that summed anything (the rest: +0)
    for (int v = wv; v < 9; v += nw) {
      if (v < 8 ? v >= 2 * nv : !nrm) continue;
      double* r = red + v * T;
      // offset 16: lanes 0-15 take warp 2 i, lanes 16-31 warp 2 i + 1
      double s[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const double* t = r + i * 64 + (lane & 16) * 2 + (lane & 15);
        s[i] = i * 64 < live ? t[0] + t[16] : 0.0;
      }
      // offsets 8, 4, 2: the lanes of either half keep one of two warps each and give the other away
#pragma unroll
      for (int h = 4; h > 0; h >>= 1) {
        const int o = 2 * h;
#pragma unroll
        for (int i = 0; i < h; ++i) {
          const bool up = lane & o;
          const double keep = up ? s[2 * i + 1] : s[2 * i], give = up ? s[2 * i] : s[2 * i + 1];
          s[i] = keep + __shfl_xor_sync(0xffffffffu, give, o);
        }
      }
      s[0] += __shfl_xor_sync(0xffffffffu, s[0], 1);
      __syncwarp();
      // the warp this lane ended with: bit 0 from lane bit 4, then bits 3, 2, 1
      if (!(lane & 1))
        r[((lane >> 4) & 1) + ((lane >> 3) & 1) * 2 + ((lane >> 2) & 1) * 4 + ((lane >> 1) & 1) * 8] = s[0];
    }
    __syncthreads();
    if (threadIdx.x < 9 && (threadIdx.x < 8 ? (int)threadIdx.x < 2 * nv : nrm)) {
      const int v = threadIdx.x;
      double x = 0.0;
#pragma unroll
      for (int u = 0; u < nw; ++u) x += red[v * T + u];
      if (v == 8) norm[blockIdx.x] = x;
      else reinterpret_cast<double*>(part + (size_t)blockIdx.x * NV + c0 + (v >> 1))[v & 1] = x;
    }
    __syncthreads();
  }
}

// h[i] = sum_g part[g * NV + i] for i in [i0, i1), every CTA in the same order.
__device__ __forceinline__ void reduce_dots(const cplx* part, int G, int i0, int i1, cplx* h) {
  const int lane = threadIdx.x & 31, wv = threadIdx.x >> 5, nw = blockDim.x >> 5;
  for (int i = i0 + wv; i < i1; i += nw) {
    double sr = 0.0, si = 0.0;
    for (int g = lane; g < G; g += 32) {
      const cplx p = __ldcg(&part[(size_t)g * NV + i]);
      sr += p.x;
      si += p.y;
    }
    sr = wsum(sr);
    si = wsum(si);
    if (lane == 0) h[i] = make_double2(sr, si);
  }
  __syncthreads();
}

// w[e] -= sum_{i in [i0, i1)} h[i] q_i[e] on the own slice
__device__ __forceinline__ void slice_project(const cplx* V, long long n, cplx* w, long long e0,
                                              int len, int i0, int i1, const cplx* h) {
  for (int e = threadIdx.x; e < len; e += blockDim.x) {
    double ax = w[e].x, ay = w[e].y;
    for (int i = i0; i < i1; ++i) {
      const cplx q = V[(size_t)i * n + e0 + e], c = h[i];
      ax = fma(-q.x, c.x, ax);
      ax = fma(q.y, c.y, ax);
      ay = fma(-q.x, c.y, ay);
      ay = fma(-q.y, c.x, ay);
    }
    w[e] = make_double2(ax, ay);
  }
  __syncthreads();
}

// partn[blockIdx.x] = ||w||^2 over the own slice (red: blockDim/32 doubles of shared memory)
__device__ __forceinline__ void slice_norm(const cplx* w, int len, double* red, double* partn) {
  double s = 0.0;
  for (int e = threadIdx.x; e < len; e += blockDim.x)
    s = fma(w[e].x, w[e].x, fma(w[e].y, w[e].y, s));
  s = wsum(s);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int v = 0; v < (int)(blockDim.x >> 5); ++v) t += red[v];
    partn[blockIdx.x] = t;
  }
}

// *dst = sum over CTAs of partn (warp 0, fixed order), visible to the CTA on return
__device__ __forceinline__ void reduce_norm(const double* partn, int G, double* dst) {
  if (threadIdx.x < 32) {
    double s = 0.0;
    for (int g = threadIdx.x; g < G; g += 32) s += __ldcg(&partn[g]);
    s = wsum(s);
    if (threadIdx.x == 0) *dst = s;
  }
  __syncthreads();
}

// Lanczos vector j done: alpha_j = Re(h1[j] + h2[j]), beta_{j+1} = sqrt(nrm2).  Warp 0 extends
// the tridiagonal T (alpha[0..j), beta[1..j] read from `alpha`, `beta`; alpha[j], beta[j+1]
// stored there when `store`) and decides whether to stop: breakdown, kcap vectors, or
// beta_{j+1} |y_j| < tol, y = exp(tau T) e_1, unless the dimension is fixed.  Where the run goes on
// for sure -- a fixed dimension not reached, or a single-precision estimate above 8 tol -- the FP64
// exponential (10-15 us of serial FP64) is left out; otherwise it decides, and lane i returns y_i
// in yr, yi when done.  Every lane returns the same done / err / breakdown, beta_{j+1} in nb and
// its reciprocal in inv.  Call from the 32 lanes of one warp.
__device__ __forceinline__ void tridiag_step(int j, double aj, double nrm2, double tr, double ti,
                                             double tol, int kcap, int fixed, double* alpha,
                                             double* beta, bool store, double& yr, double& yi,
                                             bool& done, double& err, bool& breakdown, double& nb,
                                             double& inv) {
  const int lane = threadIdx.x & 31;
  const int kk = j + 1;
  nb = sqrt(nrm2);
  inv = 1.0 / nb;
  const double a = lane < j ? alpha[lane] : (lane == j ? aj : 0.0);
  const double bl = (lane >= 1 && lane < kk) ? beta[lane] : 0.0;
  const double br = (lane + 1 < kk) ? beta[lane + 1] : 0.0;
  __syncwarp();
  if (store && lane == 0) {
    alpha[j] = aj;
    beta[j + 1] = nb;
  }
  yr = yi = err = 0.0;
  breakdown = false;
  // nb against 1e-12 of the largest entry, from the upper words first (2^-20 below their numbers)
  const int top = __reduce_max_sync(0xffffffffu, max(__double2hiint(fabs(a)), __double2hiint(fabs(bl))));
  const double low = __hiloint2double(top, 0);
  const bool clear = nb > 2e-12 * low && low > 1e-290;
  if (clear && kk < kcap) {
    if (fixed) {
      done = false;
      return;
    }
    const float e32 = lz_last_entry32((float)a, (float)bl, (float)br, kk, (float)tr, (float)ti);
    const float est = (float)nb * e32;
    if (est > 8.f * (float)tol && est < 3e38f) {
      done = false;
      return;
    }
  }
  const double scale = lz_warp_max(fmax(fabs(a), fabs(bl)));
  const double sigma = lz_exp_shifted(a, bl, br, kk, tr, ti, yr, yi);
  lz_shift_factor(sigma, tr, ti, false, yr, yi);       // modulus only: enough for the test
  const double ylr = __shfl_sync(0xffffffffu, yr, kk - 1);
  const double yli = __shfl_sync(0xffffffffu, yi, kk - 1);
  err = nb * sqrt(ylr * ylr + yli * yli);
  breakdown = nb <= 1e-12 * fmax(scale, 1e-300);
  done = breakdown || kk >= kcap || (!fixed && err < tol);
  if (done) lz_shift_factor(sigma, 0.0, ti, true, yr, yi);   // the phase, for the result
  __syncwarp();
}

}  // namespace lzc
}  // namespace tdmrg
