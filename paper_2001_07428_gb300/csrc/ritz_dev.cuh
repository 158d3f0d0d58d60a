// ritz_dev.cuh -- device routines of the Ritz solve shared by ritz.cu (one problem, one warp per
// Ritz pair) and batch.cu (many problems, one CTA each).
#pragma once

#include <math.h>

#include "common.cuh"

namespace jtr {
namespace {

// ------------------------------------------------------------------ fast path: bisection + inverse iteration
// T-bar after a thick restart has the structure (0-based, k = restart size):
//   t_ii = d_i (i < k)          kept Ritz values
//   t_ki = t_ik = b_i (i < k)   the arrow row of the Krylov-Schur form
//   t_jj = alpha_j, t_{j,j+1} = t_{j+1,j} = beta_j (k <= j < m)   Lanczos tridiagonal
// Eliminating the diagonal part first keeps this an O(m) LDL^T factorisation of T - sigma I:
//   pi_i = d_i - sigma (i < k);  pi_k = alpha_k - sigma - sum_i b_i^2 / pi_i;
//   pi_j = alpha_j - sigma - beta_{j-1}^2 / pi_{j-1} (j > k)
// and by Sylvester's law of inertia the number of negative pivots is the number of eigenvalues
// below sigma.  Each wanted eigenvalue gets one warp: FP32 multisection on this count (32 shifts
// per round), then FP64 inverse iteration with Rayleigh-quotient shifts for the eigenvector and
// eigenvalue, then an FP64 inertia check on both sides of the result.  A separate one-block
// kernel checks residuals and orthogonality; if anything fails, the Jacobi kernel recomputes all.
struct TbarView {
  const double* T;
  int ld, m, k;
  __device__ __forceinline__ double diag(int j) const { return T[(size_t)j * ld + j]; }
  __device__ __forceinline__ double arrow(int i) const { return T[(size_t)k * ld + i]; }     // i < k
  __device__ __forceinline__ double off(int j) const { return T[(size_t)(j + 1) * ld + j]; } // j >= k
};

// The count in FP32, for the multisection: d the diagonal, b2 the squares of the arrow (i < k) and of the
// off-diagonals (b2[j] of t_{j,j+1}, j >= k).  The quotients are the fast ones, good to 2 ulp, which the
// slack of the bracket covers.
__device__ __noinline__ int inertia32(const float* d, const float* b2, int k, int m, float sigma, float pivmin) {
  int neg = 0;
  float s = 0.f;
  for (int i = 0; i < k; ++i) {
    float p = d[i] - sigma;
    if (fabsf(p) < pivmin) p = -pivmin;
    neg += p < 0.f;
    s += __fdividef(b2[i], p);
  }
  float p = d[k] - sigma - s;
  if (fabsf(p) < pivmin) p = -pivmin;
  neg += p < 0.f;
  for (int j = k + 1; j < m; ++j) {
    p = d[j] - sigma - __fdividef(b2[j - 1], p);
    if (fabsf(p) < pivmin) p = -pivmin;
    neg += p < 0.f;
  }
  return neg;
}

// The tridiagonal part k .. m - 1 is eliminated from both ends at once, by two lanes: one takes k .. c
// forward, the other m - 1 .. c + 1 backward, and the last pivot joins them.  An FP64 instruction holds its
// pipe for 64 clocks whatever the active lanes, and this chain (a division an index) is most of a Ritz pair's
// time: a restart at m = 30 (this and its verification) went from 143 to 84 us with both ends at once, the two
// verification counts in one pass and FP32 copies for the multisection.
struct TwoEnds {
  int l, cnt, nf;        // this lane's end, its count, the longer (forward) count
  int j, dj;             // its first index and direction
  __device__ __forceinline__ TwoEnds(int k, int m, int end) : l(end) {
    nf = (m - k + 1) / 2;
    cnt = end ? m - k - nf : nf;
    j = end ? m - 1 : k;
    dj = end ? -1 : 1;
  }
};

// Warp-cooperative solve of (T - sigma I) x = z in place (z: right-hand side on entry, in shared
// memory); ipiv receives the reciprocal pivots.  The k eliminations of the diagonal part are
// independent and run across the lanes; the tridiagonal part goes on lanes 0 and 1, with one division an
// index and stored reciprocals elsewhere.
__device__ __noinline__ void shifted_solve_warp(const TbarView& t, double sigma, double pivmin, double* z, double* ipiv) {
  const int k = t.k, m = t.m, lane = threadIdx.x & 31;
  double s = 0.0, sr = 0.0;
  for (int i = lane; i < k; i += 32) {
    double p = t.diag(i) - sigma;
    if (fabs(p) < pivmin) p = (p < 0 ? -pivmin : pivmin);
    const double ip = 1.0 / p;
    ipiv[i] = ip;
    const double b = t.arrow(i);
    s += b * b * ip;
    sr += b * z[i] * ip;
  }
  s = warp_sum(s);
  sr = warp_sum(sr);
  if (lane < 2) {
    const TwoEnds e(k, m, lane);
    double ip = 0.0, zp = 0.0, b = 0.0;   // of the index before; b couples the two
    int j = e.j;
    for (int i = 0; i < e.cnt; ++i, j += e.dj) {
      const double l = b * ip;
      double q = t.diag(j) - sigma - b * l;
      zp = z[j] - l * zp;
      if (i == 0 && !e.l) {
        q -= s;
        zp -= sr;
      }
      z[j] = zp;
      const int c = e.l ? j - 1 : j;                       // the coupling to the next index, or across the middle
      if (c >= k && c + 1 < m) b = t.off(c);
      if (i + 1 < e.cnt || !e.l) {                         // the backward end's last pivot is the joined one
        if (fabs(q) < pivmin) q = (q < 0 ? -pivmin : pivmin);
        ip = 1.0 / q;
        ipiv[j] = ip;
      } else {
        ip = q;                                            // carried to the join
      }
    }
    // join: x_{c+1} = (z_{c+1} - b z_c / q_c) / (q_{c+1} - b^2 / q_c), x_c = (z_c - b x_{c+1}) / q_c
    const double ipc = __shfl_sync(3u, ip, 0), zc = __shfl_sync(3u, zp, 0), bc = __shfl_sync(3u, b, 0);
    const double qe = __shfl_sync(3u, ip, 1), ze = __shfl_sync(3u, zp, 1);
    double zn;
    if (m - k > 1) {
      const double l = bc * ipc;
      double q = qe - bc * l;
      if (fabs(q) < pivmin) q = (q < 0 ? -pivmin : pivmin);
      const double xe = (ze - l * zc) / q;
      zn = lane ? xe : (zc - bc * xe) * ipc;
    } else {
      zn = zc * ipc;
    }
    j -= e.dj;                                             // this end's last index
    if (e.cnt > 0) z[j] = zn;
    for (int i = 1; i < e.cnt; ++i) {
      const double o = t.off(e.l ? j : j - 1);
      j -= e.dj;
      zn = (z[j] - o * zn) * ipiv[j];
      z[j] = zn;
    }
  }
  __syncwarp();
  const double zk = z[k];
  for (int i = lane; i < k; i += 32) z[i] = (z[i] - t.arrow(i) * zk) * ipiv[i];
  __syncwarp();
}

// Warp-cooperative FP64 inertia counts of T - sigma I for two shifts (lanes 0 .. 15 and 16 .. 31 take one
// each), the elimination as above.  Lane 0 returns the count of s0 and lane 16 that of s1.
__device__ __noinline__ int inertia2_warp(const TbarView& t, double s0, double s1, double pivmin) {
  const int k = t.k, m = t.m, lane = threadIdx.x & 31, sub = lane & 15;
  const double sigma = lane < 16 ? s0 : s1;
  double s = 0.0;
  int neg = 0;
  for (int i = sub; i < k; i += 16) {
    double p = t.diag(i) - sigma;
    if (fabs(p) < pivmin) p = -pivmin;
    neg += p < 0;
    const double b = t.arrow(i);
    s += b * b / p;
  }
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) {
    s += __shfl_xor_sync(0xffffffffu, s, o);
    neg += __shfl_xor_sync(0xffffffffu, neg, o);
  }
  if (sub) neg = 0;
  double p = 0.0, r = 0.0;   // the pivot; what it takes from the next one
  if (sub < 2) {
    const TwoEnds e(k, m, sub);
    int j = e.j;
    for (int i = 0; i < e.cnt; ++i, j += e.dj) {
      p = t.diag(j) - sigma - r;
      if (i == 0 && !e.l) p -= s;
      if (i + 1 < e.cnt || !e.l) {
        if (fabs(p) < pivmin) p = -pivmin;
        neg += p < 0;
        const int c = e.l ? j - 1 : j;
        if (c + 1 < m) {
          const double b = t.off(c);
          r = b * b / p;
        }
      }
    }
  }
  const double rc = __shfl_xor_sync(0xffffffffu, r, 1);
  if (sub == 1 && m - k > 1) {   // the joined pivot
    p -= rc;
    if (fabs(p) < pivmin) p = -pivmin;
    neg += p < 0;
  }
  return neg + __shfl_xor_sync(0xffffffffu, neg, 1);
}

__device__ double warp_normalize(double* z, int m) {
  const int lane = threadIdx.x & 31;
  double s = 0.0;
  for (int i = lane; i < m; i += 32) s += z[i] * z[i];
  s = warp_sum(s);
  const double inv = 1.0 / sqrt(s);
  __syncwarp();
  for (int i = lane; i < m; i += 32) z[i] *= inv;
  __syncwarp();
  return s;
}

// (T z)_i for all i, lane-parallel, into tz.
__device__ void warp_apply(const TbarView& t, const double* z, double* tz) {
  const int lane = threadIdx.x & 31, k = t.k, m = t.m;
  for (int i = lane; i < m; i += 32) {
    double v;
    if (i < k) {
      v = t.diag(i) * z[i] + t.arrow(i) * z[k];
    } else {
      v = t.diag(i) * z[i];
      if (i == k) {
        for (int q = 0; q < k; ++q) v += t.arrow(q) * z[q];
      } else {
        v += t.off(i - 1) * z[i - 1];
      }
      if (i + 1 < m) v += t.off(i) * z[i + 1];
    }
    tz[i] = v;
  }
  __syncwarp();
}

// One warp computes the eigenpair of index r (ascending order) of the T-bar held in T (ld ldt, m x m,
// restart size k): FP32 multisection on the inertia count, FP64 inverse iteration with Rayleigh-
// quotient shifts, and an FP64 inertia check on both sides.  z, piv, tz: warp-private scratch of m
// doubles each.  Writes the normalised eigenvector to zout (m doubles) and returns the eigenvalue,
// or NaN if the inertia check fails.
__device__ double ritz_pair_warp(const double* T, int ldt, int m, int k, int r, double* z, double* piv, double* tz,
                                 double* zout) {
  const int lane = threadIdx.x & 31;
  const TbarView t{T, ldt, m, k};
  // Gershgorin interval and scale
  double glo = 1e300, ghi = -1e300;
  for (int j = lane; j < m; j += 32) {
    double rad = 0.0;
    if (j < k) rad = fabs(t.arrow(j));
    else {
      if (j == k) for (int q = 0; q < k; ++q) rad += fabs(t.arrow(q));
      else rad += fabs(t.off(j - 1));
      if (j + 1 < m) rad += fabs(t.off(j));
    }
    glo = fmin(glo, t.diag(j) - rad);
    ghi = fmax(ghi, t.diag(j) + rad);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    glo = fmin(glo, __shfl_xor_sync(0xffffffffu, glo, o));
    ghi = fmax(ghi, __shfl_xor_sync(0xffffffffu, ghi, o));
  }
  const double tnorm = fmax(fabs(glo), fabs(ghi));
  glo -= 1e-6 * tnorm + 1e-300;
  ghi += 1e-6 * tnorm + 1e-300;
  // FP32 multisection: 32 shifts per round, keep [lo, hi] with count(lo) <= r < count(hi)
  float lo = (float)glo, hi = (float)ghi;
  const float pmin32 = (float)(tnorm * 1e-30) + 1e-30f;
  float* d32 = (float*)piv;                      // FP32 copies: a conversion costs as much as an FP64 instruction
  float* b32 = (float*)tz;
  for (int j = lane; j < m; j += 32) {
    d32[j] = (float)t.diag(j);
    const float b = j < k ? (float)t.arrow(j) : j + 1 < m ? (float)t.off(j) : 0.f;
    b32[j] = b * b;
  }
  __syncwarp();
  for (int round = 0; round < 8; ++round) {
    const float w = (hi - lo) / 33.0f;
    const float sig = lo + w * (float)(lane + 1);
    const int cnt = inertia32(d32, b32, k, m, sig, pmin32);
    const unsigned below = __ballot_sync(0xffffffffu, cnt <= r);   // shifts still at or below lambda_r
    const int nb = __popc(below);                                   // counts are monotone in the shift
    const float nlo = nb > 0 ? __shfl_sync(0xffffffffu, sig, nb - 1) : lo;
    const float nhi = nb < 32 ? __shfl_sync(0xffffffffu, sig, nb) : hi;
    lo = nlo;
    hi = nhi;
    if (hi - lo <= 4.0f * 1.2e-7f * fmaxf(fabsf(lo), fabsf(hi))) break;
  }
  const double lo64 = (double)lo, hi64 = (double)hi;
  const double slack = 1e-6 * tnorm;             // FP32 rounding of T moves eigenvalues by ~6e-8 ||T||
  double sigma = 0.5 * (lo64 + hi64);
  const double pivmin = 1e-18 * tnorm + 1e-300;
  // FP64 inverse iteration from a fixed pseudo-random start, four solves, each followed by a
  // Rayleigh quotient that becomes the next shift (kept only while inside the FP32 bracket).  With three,
  // what was left of neighbours at a relative gap of 1e-4 showed: ||x|| - 1 and x^H A x - lambda of late
  // pairs at 16^4 came out between 1e-13 and 8e-11 as rounding fell; with four they stay below 4e-13
  for (int j = lane; j < m; j += 32) z[j] = u01_sym(0x9E37ull * (uint64_t)(r + 1) + (uint64_t)j) + 0.5;
  __syncwarp();
  warp_normalize(z, m);
  double lambda = sigma;
  for (int it = 0; it < 4; ++it) {
    shifted_solve_warp(t, sigma, pivmin, z, piv);
    warp_normalize(z, m);
    warp_apply(t, z, tz);
    double q = 0.0;
    for (int j = lane; j < m; j += 32) q += z[j] * tz[j];
    lambda = warp_sum(q);
    if (lambda >= lo64 - slack && lambda <= hi64 + slack) sigma = lambda;
  }
  // FP64 inertia on both sides: lambda must be the r-th eigenvalue (Sylvester)
  const double delta = 1e-9 * tnorm;
  const int cnt2 = inertia2_warp(t, lambda - delta, lambda + delta, pivmin);
  const int c_lo = __shfl_sync(0xffffffffu, cnt2, 0), c_hi = __shfl_sync(0xffffffffu, cnt2, 16);
  for (int j = lane; j < m; j += 32) zout[j] = z[j];
  return (c_lo <= r && c_hi >= r + 1 && lambda == lambda) ? lambda : NAN;
}

}  // namespace
}  // namespace jtr
