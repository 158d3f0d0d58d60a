// ritz.cu -- the restart of Algorithm 1 on the device: Rayleigh-Ritz solve of T_m, the basis
// rotation V_m := V_m Z_m (Corollary 2 keeps V and W = J V^* orthogonal under it), the shrink to
// k + 1 vectors with v_{k+1} = v_{m+1}, and the output gather with partners y = J x^* (eq. (2)).
#include "fixed.cuh"
#include "internal.h"
#include "ritz_dev.cuh"
#include "../../include/jtrlan.h"

namespace jtr {

namespace {

// ------------------------------------------------------------------ cyclic Jacobi, one CTA
// T_m = Z Lambda Z^T for the real symmetric m x m leading block of T-bar (arrowhead plus
// tridiagonal).  Parallel Jacobi: each round applies mp/2 disjoint plane rotations chosen by the
// round-robin ordering (player 0 fixed, the others rotate), so a sweep of mp-1 rounds visits every
// pair once.  Rotation angles follow Rutishauser's stable formulas (Golub & Van Loan, sym.schur2).
// An odd m is padded with one decoupled index.  Sweeps stop when no off-diagonal entry exceeds
// 1e-17 (|a_pp| + |a_qq|) -- i.e. T is diagonal to working precision -- or after 60 sweeps.
constexpr int kRitzThreads = 1024;
constexpr int kMaxPairs = 512;

__global__ void __launch_bounds__(kRitzThreads)
ritz_jacobi_kernel(const double* __restrict__ T, int ldt, int m, int which, double* __restrict__ lam,
                   double* __restrict__ Zout, double* __restrict__ work, int use_smem, const int* __restrict__ gate,
                   long long* __restrict__ fallbacks) {
  extern __shared__ double dsm[];
  if (gate && *gate == 0) return;   // the fast path succeeded
  if (fallbacks && threadIdx.x == 0) *fallbacks += 1;
  __shared__ double rc[kMaxPairs], rs[kMaxPairs], rt[kMaxPairs], rapp[kMaxPairs], raqq[kMaxPairs],
      rapq[kMaxPairs];
  __shared__ int rp[kMaxPairs], rq[kMaxPairs];
  __shared__ int s_rot;
  __shared__ int rank_of[2 * kMaxPairs];
  const int mp = m + (m & 1);
  const int half = mp / 2;
  double* A = use_smem ? dsm : work;
  double* Z = A + (size_t)mp * mp;
  const int tid = threadIdx.x;
  for (int e = tid; e < mp * mp; e += kRitzThreads) {
    const int r = e / mp, c = e % mp;
    A[e] = (r < m && c < m) ? T[(size_t)r * ldt + c] : 0.0;
    Z[e] = (r == c) ? 1.0 : 0.0;
  }
  __syncthreads();
  for (int sweep = 0; sweep < 60; ++sweep) {
    if (tid == 0) s_rot = 0;
    __syncthreads();
    for (int round = 0; round < mp - 1; ++round) {
      for (int k = tid; k < half; k += kRitzThreads) {
        // round-robin pairing: position 0 holds player 0, positions 1..mp-1 rotate
        const int a = (k == 0) ? 0 : ((k - 1 + round) % (mp - 1)) + 1;
        const int b = ((mp - 2 - k + round) % (mp - 1)) + 1;
        const int p = min(a, b), q = max(a, b);
        const double app = A[p * mp + p], aqq = A[q * mp + q], apq = A[p * mp + q];
        double c = 1.0, s = 0.0, t = 0.0;
        if (fabs(apq) > 1e-17 * (fabs(app) + fabs(aqq)) && fabs(apq) > 1e-300) {
          const double tau = (aqq - app) / (2.0 * apq);
          t = (tau >= 0.0 ? 1.0 : -1.0) / (fabs(tau) + sqrt(1.0 + tau * tau));
          c = 1.0 / sqrt(1.0 + t * t);
          s = t * c;
          s_rot = 1;
        }
        rp[k] = p; rq[k] = q; rc[k] = c; rs[k] = s; rt[k] = t;
        rapp[k] = app; raqq[k] = aqq; rapq[k] = apq;
      }
      __syncthreads();
      // rows p, q  <-  J^T A
      for (int e = tid; e < half * mp; e += kRitzThreads) {
        const int k = e / mp, l = e % mp;
        if (rs[k] == 0.0) continue;
        const int p = rp[k], q = rq[k];
        const double c = rc[k], s = rs[k];
        const double ap = A[p * mp + l], aq = A[q * mp + l];
        A[p * mp + l] = c * ap - s * aq;
        A[q * mp + l] = s * ap + c * aq;
      }
      __syncthreads();
      // columns p, q  <-  A J,  Z <- Z J
      for (int e = tid; e < half * mp; e += kRitzThreads) {
        const int k = e / mp, l = e % mp;
        if (rs[k] == 0.0) continue;
        const int p = rp[k], q = rq[k];
        const double c = rc[k], s = rs[k];
        const double ap = A[l * mp + p], aq = A[l * mp + q];
        A[l * mp + p] = c * ap - s * aq;
        A[l * mp + q] = s * ap + c * aq;
        const double zp = Z[l * mp + p], zq = Z[l * mp + q];
        Z[l * mp + p] = c * zp - s * zq;
        Z[l * mp + q] = s * zp + c * zq;
      }
      __syncthreads();
      for (int k = tid; k < half; k += kRitzThreads) {
        if (rs[k] == 0.0) continue;
        const int p = rp[k], q = rq[k];
        A[p * mp + q] = 0.0;
        A[q * mp + p] = 0.0;
        A[p * mp + p] = rapp[k] - rt[k] * rapq[k];
        A[q * mp + q] = raqq[k] + rt[k] * rapq[k];
      }
      __syncthreads();
    }
    if (!s_rot) break;
    __syncthreads();
  }
  // sort the m eigenvalues toward the wanted end (stable in the index)
  for (int i = tid; i < m; i += kRitzThreads) {
    const double li = A[i * mp + i];
    int r = 0;
    for (int k = 0; k < m; ++k) {
      const double lk = A[k * mp + k];
      const bool before = (which == JTRLAN_LARGEST) ? (lk > li) : (lk < li);
      if (before || (lk == li && k < i)) ++r;
    }
    rank_of[r] = i;
  }
  __syncthreads();
  for (int r = tid; r < m; r += kRitzThreads) lam[r] = A[rank_of[r] * mp + rank_of[r]];
  for (int e = tid; e < m * m; e += kRitzThreads) {
    const int c = e / m, l = e % m;  // Zout column-major: component l of eigenvector c
    Zout[(size_t)c * m + l] = Z[l * mp + rank_of[c]];
  }
}

constexpr int kBisectWarps = 4;

__global__ void __launch_bounds__(32 * kBisectWarps)
ritz_bisect_kernel(const double* __restrict__ T, int ldt, int m, int k, int kk, int which, double* __restrict__ lam,
                   double* __restrict__ Zout, int* __restrict__ ok) {
  extern __shared__ double rsm[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int i = blockIdx.x * kBisectWarps + warp;
  if (i >= kk) return;
  double* z = rsm + (size_t)warp * 3 * m;
  const int r = (which == JTRLAN_LARGEST) ? m - 1 - i : i;   // index in ascending order
  const double lambda = ritz_pair_warp(T, ldt, m, k, r, z, z + m, z + 2 * m, Zout + (size_t)i * m);
  if (lane == 0) {
    lam[i] = lambda;
    ok[i] = (lambda == lambda) ? 1 : 0;
  }
}

// One block: residual ||T z_i - lambda_i z_i||, orthogonality of neighbours, the per-pair inertia
// flags; sets *fallback (read by the Jacobi kernel).
__global__ void __launch_bounds__(256)
ritz_check_kernel(const double* __restrict__ T, int ldt, int m, int k, int kk, int which, const double* __restrict__ lam,
                  const double* __restrict__ Z, const int* __restrict__ ok, int* __restrict__ fallback) {
  __shared__ int bad;
  if (threadIdx.x == 0) bad = 0;
  __syncthreads();
  const TbarView t{T, ldt, m, k};
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  double tn = 0.0;
  for (int j = 0; j < m; ++j) tn = fmax(tn, fabs(t.diag(j)));
  for (int i = warp; i < kk; i += 8) {
    const double* z = Z + (size_t)i * m;
    double res = 0.0, dot = 0.0, nn = 0.0;
    for (int j = lane; j < m; j += 32) {
      double v = t.diag(j) * z[j];
      if (j < k) v += t.arrow(j) * z[k];
      else {
        if (j == k) for (int q = 0; q < k; ++q) v += t.arrow(q) * z[q];
        else v += t.off(j - 1) * z[j - 1];
        if (j + 1 < m) v += t.off(j) * z[j + 1];
      }
      v -= lam[i] * z[j];
      res += v * v;
      nn += z[j] * z[j];
      if (i + 1 < kk) dot += z[j] * Z[(size_t)(i + 1) * m + j];
    }
    res = warp_sum(res); dot = warp_sum(dot); nn = warp_sum(nn);
    if (lane == 0) {
      bool good = ok[i] && sqrt(res) <= 1e-11 * fmax(tn, 1e-300) && fabs(nn - 1.0) <= 1e-12 && fabs(dot) <= 1e-9;
      if (i + 1 < kk) good = good && ((which == JTRLAN_LARGEST) ? lam[i] > lam[i + 1] : lam[i] < lam[i + 1]);
      if (!good) atomicExch(&bad, 1);
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) *fallback = bad;
}

// ------------------------------------------------------------------ rotation V_m Z
// out (n x kk complex) = V Z for the fixed-point basis (fixed.cuh), Z real: exact integer sums of two-limb
// products, 7.5 a clock and SM against 2 FP64 multiply-adds.  A lane owns a complex row and four columns
// of Z (8 sums); the warps of a block share the row's loads through L1 and take other columns.  Z, scaled
// by the columns' 2^e and converted on the scale of its largest entry per column, passes through shared
// memory 64 rows at a time, the number of products a sum holds; then the sums leave for FP64.
// A column of Z that is a unit vector (a locked pair's) copies that column of V to the last bit.
// 8^4 (m 60): 58 us a launch, 199 us in FP64.
constexpr int kRotK = 64, kRotC = 4, kRotGroups = 8;

__global__ void __launch_bounds__(32 * kRotGroups)
rotate_fx_kernel(const fxc* __restrict__ V, const int* __restrict__ vexp, int64_t n, int m, const double* __restrict__ Z,
                 int kk, double2* __restrict__ out) {
  __shared__ __align__(16) int2 zs[kRotK][kRotC * kRotGroups];
  __shared__ int zk[kRotC * kRotGroups], zunit[kRotC * kRotGroups];   // K; k (or ~k for -1) of a unit column, else m
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, cols = kRotC * (blockDim.x >> 5);
  const int c0 = blockIdx.y * cols;
  const int64_t p = (int64_t)blockIdx.x * 32 + lane;
  for (int c = w; c < cols; c += blockDim.x >> 5) {     // K of each scaled column of Z
    int f = 0, cnt = 0, unit = m;
    if (c0 + c < kk)
      for (int k = lane; k < m; k += 32) {
        const double z = Z[(int64_t)(c0 + c) * m + k];
        const int g = fx_field(z);
        f = max(f, g ? max(g + vexp[k] - 1023, 1) : 0);
        if (g >= 1023 - 60) {
          ++cnt;
          unit = __double2hiint(z) < 0 ? ~k : k;
        }
      }
    f = __reduce_max_sync(0xffffffffu, f);
    cnt = __reduce_add_sync(0xffffffffu, cnt);
    const unsigned has = __ballot_sync(0xffffffffu, unit != m);
    if (has) unit = __shfl_sync(0xffffffffu, unit, __ffs(has) - 1);
    if (lane == 0) {
      zk[c] = f + 1;
      zunit[c] = cnt == 1 ? unit : m;
    }
  }
  double2 o[kRotC];
#pragma unroll
  for (int c = 0; c < kRotC; ++c) o[c] = make_double2(0.0, 0.0);
  for (int k0 = 0; k0 < m; k0 += kRotK) {
    const int kn = min(kRotK, m - k0);
    __syncthreads();
    for (int e = threadIdx.x; e < cols * kRotK; e += blockDim.x) {
      const int k = e % kRotK, c = e / kRotK;
      int2 v = make_int2(0, 0);
      if (k < kn && c0 + c < kk) {
        const fx2 t = fx_limbs<true>(Z[(int64_t)(c0 + c) * m + k0 + k], zk[c] - (vexp[k0 + k] - 1023));
        v = make_int2(t.h, t.l);
      }
      zs[k][c] = v;
    }
    __syncthreads();
    FxAcc a[kRotC][2];
#pragma unroll
    for (int c = 0; c < kRotC; ++c) {
      fx_zero(a[c][0]);
      fx_zero(a[c][1]);
    }
    if (p < n) {
      const fxc* v = V + (int64_t)k0 * n + p;
      auto mac = [&](fxc x, int k) {
        const fx2 re = fx_round(x.re), im = fx_round(x.im);
#pragma unroll
        for (int c = 0; c < kRotC; c += 2) {
          const int4 z = *reinterpret_cast<const int4*>(&zs[k][kRotC * w + c]);
          fx_mac(a[c][0], re, fx2{z.x, z.y});
          fx_mac(a[c][1], im, fx2{z.x, z.y});
          fx_mac(a[c + 1][0], re, fx2{z.z, z.w});
          fx_mac(a[c + 1][1], im, fx2{z.z, z.w});
        }
      };
      int k = 0;
      for (; k + 3 < kn; k += 4) {
        fxc x[4];
#pragma unroll
        for (int t = 0; t < 4; ++t) x[t] = v[(int64_t)(k + t) * n];
#pragma unroll
        for (int t = 0; t < 4; ++t) mac(x[t], k + t);
      }
      for (; k < kn; ++k) mac(v[(int64_t)k * n], k);
    }
#pragma unroll
    for (int c = 0; c < kRotC; ++c) {
      const int K = zk[kRotC * w + c];
      const double re = fx_lane_value(a[c][0], K), im = fx_lane_value(a[c][1], K);
      if (k0 == 0) o[c] = make_double2(re, im);
      else o[c] = make_double2(o[c].x + re, o[c].y + im);
    }
  }
  if (p < n)
#pragma unroll
    for (int c = 0; c < kRotC; ++c) {
      const int u = zunit[kRotC * w + c], k = u < 0 ? ~u : u;
      if (k < m) {
        const fxc x = V[(int64_t)k * n + p];
        const double re = fx_load(x.re, vexp[k]), im = fx_load(x.im, vexp[k]);
        o[c] = u < 0 ? make_double2(-re, -im) : make_double2(re, im);
      }
      if (c0 + kRotC * w + c < kk) out[(int64_t)(c0 + kRotC * w + c) * n + p] = o[c];
    }
}

// FP32 rotation for the mixed-precision phase: Z rounded to FP32, FP32 accumulation.
__global__ void __launch_bounds__(256)
rotate32_kernel(const float* __restrict__ V, int64_t rows, int m, const double* __restrict__ Z, int kk,
                float* __restrict__ out) {
  constexpr int BM = 128, BN = 32, BK = 16;
  __shared__ float As[BK][BM];
  __shared__ float Bs[BK][BN];
  const int tid = threadIdx.x;
  const int64_t row0 = (int64_t)blockIdx.x * BM;
  const int col0 = blockIdx.y * BN;
  const int tr = tid % 32, tc = tid / 32;  // rows tr + 32 i (i < 4), cols tc + 8 j (j < 4)
  float acc[4][4] = {};
  for (int k0 = 0; k0 < m; k0 += BK) {
    for (int e = tid; e < BK * BM; e += 256) {
      const int kx = e / BM, r = e % BM;
      const int64_t gr = row0 + r;
      As[kx][r] = (gr < rows && k0 + kx < m) ? V[(int64_t)(k0 + kx) * rows + gr] : 0.f;
    }
    for (int e = tid; e < BK * BN; e += 256) {
      const int kx = e / BN, c = e % BN;
      Bs[kx][c] = (k0 + kx < m && col0 + c < kk) ? (float)Z[(int64_t)(col0 + c) * m + k0 + kx] : 0.f;
    }
    __syncthreads();
#pragma unroll
    for (int x = 0; x < BK; ++x) {
      float a[4], b[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) a[i] = As[x][tr + 32 * i];
#pragma unroll
      for (int j = 0; j < 4; ++j) b[j] = Bs[x][tc + 8 * j];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int64_t gr = row0 + tr + 32 * i;
    if (gr >= rows) continue;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int gc = col0 + tc + 8 * j;
      if (gc < kk) out[(int64_t)gc * rows + gr] = acc[i][j];
    }
  }
}

template <typename R>
__global__ void shrink_kernel(cplx<R>* V, const cplx<R>* Vsrc, int64_t n, const int* perm, int k, int m) {
  const int c = blockIdx.y;
  const cplx<R>* src = (c < k) ? Vsrc + (int64_t)perm[c] * n : V + (int64_t)m * n;
  cplx<R>* dst = V + (int64_t)c * n;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    dst[i] = src[i];
}

__global__ void reduce_norms_kernel(const double* part, int nblk, double* out) {
  __shared__ double sh[32];
  const int c = blockIdx.x;
  double s = 0.0;
  for (int b = threadIdx.x; b < nblk; b += blockDim.x) s += part[(int64_t)c * nblk + b];
  s = block_sum(s, sh);
  if (threadIdx.x == 0) out[c] = sqrt(s);
}

__global__ void report_kernel(const double* lam, const double* Z, int m, const double* T, int ldt,
                              const StepState* st, double* rep) {
  for (int i = threadIdx.x; i < m; i += blockDim.x) {
    rep[i] = lam[i];
    rep[m + i] = Z[(int64_t)i * m + (m - 1)];   // z_{m,i}: last component of eigenvector i
  }
  if (threadIdx.x == 0) {
    rep[2 * m] = T[(int64_t)m * ldt + m - 1];    // t_{m+1,m} = beta_m
    rep[2 * m + 1] = (double)st->status;
    rep[2 * m + 2] = (double)st->n_passes;
    rep[2 * m + 3] = st->tmax;
    rep[2 * m + 4] = st->units_first;
    rep[2 * m + 5] = st->units_dot;
    rep[2 * m + 6] = st->units_update;
    rep[2 * m + 7] = (double)st->n_ritz_fallbacks;
  }
}

inline int grid_for(int64_t n) {
  int64_t g = (n + 255) / 256;
  return (int)(g > 1216 ? 1216 : (g < 1 ? 1 : g));
}

}  // namespace

cudaError_t launch_ritz(const double* T, int ldt, int m, int k, int kk, int which, double* lam, double* Z,
                        int* flags, cudaStream_t s) {
  if (m < 1 || m > 2 * kMaxPairs - 1 || k < 0 || k >= m || kk < 1 || kk > m) return cudaErrorInvalidValue;
  int* ok = flags + 1;        // kk per-pair flags
  int* fallback = flags;      // 1: run the Jacobi kernel
  const size_t bsm = (size_t)kBisectWarps * 3 * m * sizeof(double);
  if (bsm > 48 * 1024) {
    cudaError_t e = allow_dyn_smem((const void*)ritz_bisect_kernel, (size_t)bsm);
    if (e != cudaSuccess) return e;
  }
  ritz_bisect_kernel<<<(kk + kBisectWarps - 1) / kBisectWarps, 32 * kBisectWarps, bsm, s>>>(T, ldt, m, k, kk, which, lam,
                                                                                            Z, ok);
  ritz_check_kernel<<<1, 256, 0, s>>>(T, ldt, m, k, kk, which, lam, Z, ok, fallback);
  return cudaGetLastError();
}

static cudaError_t jacobi_launch(const double* T, int ldt, int m, int which, double* lam, double* Z, double* work,
                                 const int* gate, long long* fallbacks, cudaStream_t s) {
  if (m < 1 || m > 2 * kMaxPairs - 1) return cudaErrorInvalidValue;
  const int mp = m + (m & 1);
  const size_t bytes = (size_t)2 * mp * mp * sizeof(double);
  const int use_smem = bytes <= 160 * 1024;
  if (use_smem) {
    cudaError_t e = allow_dyn_smem((const void*)ritz_jacobi_kernel, (size_t)bytes);
    if (e != cudaSuccess) return e;
  }
  ritz_jacobi_kernel<<<1, kRitzThreads, use_smem ? bytes : 0, s>>>(T, ldt, m, which, lam, Z, work, use_smem, gate,
                                                                   fallbacks);
  return cudaGetLastError();
}

cudaError_t launch_ritz_fallback(const double* T, int ldt, int m, int which, double* lam, double* Z, double* work,
                                 const int* flags, long long* fallbacks, cudaStream_t s) {
  return jacobi_launch(T, ldt, m, which, lam, Z, work, flags, fallbacks, s);
}

cudaError_t launch_ritz_jacobi(const double* T, int ldt, int m, int which, double* lam, double* Z, double* work,
                               cudaStream_t s) {
  return jacobi_launch(T, ldt, m, which, lam, Z, work, nullptr, nullptr, s);
}

template <>
cudaError_t launch_rotate<float>(const void* V, int64_t n, int m, const double* Z, int kk, void* Vout, cudaStream_t s) {
  const int64_t rows = 2 * n;
  dim3 grid((unsigned)((rows + 127) / 128), (unsigned)((kk + 31) / 32));
  rotate32_kernel<<<grid, 256, 0, s>>>((const float*)V, rows, m, Z, kk, (float*)Vout);
  return cudaGetLastError();
}

cudaError_t launch_rotate_fx(const void* V, const int* vexp, int64_t n, int m, const double* Z, int kk, void* out,
                             cudaStream_t s) {
  const int need = (kk + kRotC - 1) / kRotC;                       // column groups
  const int tiles = (need + kRotGroups - 1) / kRotGroups;
  const int groups = (need + tiles - 1) / tiles;                   // a block's, evenly filled
  rotate_fx_kernel<<<dim3((unsigned)((n + 31) / 32), (unsigned)tiles), 32 * groups, 0, s>>>(
      (const fxc*)V, vexp, n, m, Z, kk, (double2*)out);
  return cudaGetLastError();
}

template <typename R>
cudaError_t launch_shrink(void* V, const void* Vsrc, int64_t n, const int* perm, int k, int m, cudaStream_t s) {
  dim3 grid(grid_for(n) / 4 + 1, k + 1);
  shrink_kernel<R><<<grid, 256, 0, s>>>((cplx<R>*)V, (const cplx<R>*)Vsrc, n, perm, k, m);
  return cudaGetLastError();
}

cudaError_t launch_reduce_norms(const double* part, int nblk, int ncol, double* out, cudaStream_t s) {
  if (ncol <= 0) return cudaSuccess;
  reduce_norms_kernel<<<ncol, 128, 0, s>>>(part, nblk, out);
  return cudaGetLastError();
}

cudaError_t launch_report(const double* lam, const double* Z, int m, const double* T, int ldt, const StepState* st,
                          double* rep, cudaStream_t s) {
  report_kernel<<<1, 256, 0, s>>>(lam, Z, m, T, ldt, st, rep);
  return cudaGetLastError();
}

template cudaError_t launch_shrink<float>(void*, const void*, int64_t, const int*, int, int, cudaStream_t);

}  // namespace jtr
