// gsfx.cu -- the Gram-Schmidt part of the Lanczos step with J-symmetry (Algorithm 2) on the fixed-point
// basis (fixed.cuh) of plain FP64; the method and the formulas of c_v, c_w and the update are those at the
// head of gs.cu, whose kernels serve FP32.
//
// On this GPU FP64 multiply-adds run at 2 a clock and SM, so projections in plain FP64 are bound by that
// pipe, not by the read of V.  Here
//   * the inner products c_v = V^H y, c_w = W^H y are exact integer sums of two-limb numbers, 3.75 times
//     the FP64 rate (four wide multiply-adds a product, 30 a clock and SM); y is converted once per row block into shared memory on that block's largest entry;
//   * the update y -= V c_v + W c_w splits the columns: those whose coefficients are not small (in a
//     Lanczos step beta_{j-1}'s, and the arrow's right after a restart) are applied in the same exact
//     sums, the others, of rounding size, by their leading 28 bits in one integer sum (see UpdFx);
//   * sums of per-block partials are integer too: an FP64 instruction holds its SM quarter's pipe for 64
//     clocks whatever its lanes do, and with FP64 adds in every warp of every block one norm took 7,000.
// y, alpha, beta, the norms and the test stay in FP64.
#include <cooperative_groups.h>

#include "fixed.cuh"
#include "internal.h"

namespace jtr {

namespace {

constexpr int kT = 512, kW = kT / 32;
constexpr int kChunk = 512;        // row pairs converted at a time: 16 a lane, 64 products per sum
constexpr double kSqrt2 = 1.4142135623730951;
constexpr int kClusterMax = 8;

// ------------------------------------------------------------------ inner products
// Rows [r0, r0 + rows) of y (rows <= kChunk) as limbs into ys ([2][rows]: h_re, l_re, h_im, l_im);
// returns their K.  With SubAlpha y is first replaced by y - alpha v_j, and *nrm grows by |y|^2.
template <bool SubAlpha>
__device__ int load_chunk(const GSArgs& a, int64_t r0, int rows, int4* ys, int* smax, double alpha, double* nrm) {
  double2* y = (double2*)a.y;
  const double2* vj = a.x;
  constexpr int NR = 2 * kChunk / kT;                // entry e: row e of the first half, then of the second
  double2 v[NR];
  int ex = 0;
#pragma unroll
  for (int u = 0; u < NR; ++u) {
    const int e = threadIdx.x + u * kT;
    v[u] = make_double2(0.0, 0.0);
    if (e < 2 * rows) {
      const int64_t i = r0 + (e < rows ? e : e - rows + a.h);
      double2 t = y[i];
      if (SubAlpha) {
        const double2 w = vj[i];
        t.x -= alpha * w.x;
        t.y -= alpha * w.y;
        y[i] = t;
        *nrm += cabs2(t);
      }
      v[u] = t;
      ex = max(ex, max(fx_field(t.x), fx_field(t.y)));
    }
  }
  ex = __reduce_max_sync(0xffffffffu, ex);
  __syncthreads();                                   // the last chunk's readers of ys and smax are done
  if ((threadIdx.x & 31) == 0) smax[threadIdx.x >> 5] = ex;
  __syncthreads();
#pragma unroll
  for (int w = 0; w < kW; ++w) ex = max(ex, smax[w]);
  const int K = ex + 1;
#pragma unroll
  for (int u = 0; u < NR; ++u) {
    const int e = threadIdx.x + u * kT;
    if (e < 2 * rows) {
      const fx2 re = fx_limbs<true>(v[u].x, K), im = fx_limbs<true>(v[u].y, K);
      ys[e] = make_int4(re.h, re.l, im.h, im.l);
    }
  }
  __syncthreads();
  return K;
}

// The 16 products of one row pair, c_v += conj(v1) y1 + conj(v2) y2 and c_w += v1 y2 - v2 y1, into seven
// sums: Re c_v = s0, Im c_v = s1 - s2, Re c_w = s3 - s4, Im c_w = s5 - s6.  (With the signs on the factors
// instead, the multiply-add pipe, which is the bound here, also ran about 25 negations and moves a row.)
__device__ __forceinline__ void dot_row(FxAcc* s, fxc v1, fxc v2, int4 w1, int4 w2) {
  const fx2 y1x{w1.x, w1.y}, y1y{w1.z, w1.w}, y2x{w2.x, w2.y}, y2y{w2.z, w2.w};
  const fx2 a = fx_round(v1.re), b = fx_round(v1.im), c = fx_round(v2.re), d = fx_round(v2.im);
  fx_mac(s[0], a, y1x); fx_mac(s[0], b, y1y); fx_mac(s[0], c, y2x); fx_mac(s[0], d, y2y);
  fx_mac(s[1], a, y1y); fx_mac(s[1], c, y2y); fx_mac(s[2], b, y1x); fx_mac(s[2], d, y2x);
  fx_mac(s[3], a, y2x); fx_mac(s[3], d, y1y); fx_mac(s[4], b, y2y); fx_mac(s[4], c, y1x);
  fx_mac(s[5], a, y2y); fx_mac(s[5], b, y2x); fx_mac(s[6], c, y1y); fx_mac(s[6], d, y1x);
}

// Partials of c_v and c_w of columns 0..j over one chunk: warp q takes columns q, q + kW, ..., two 32-row
// steps' loads at a time; the sums of eight of its columns are kept one a lane and leave for FP64
// together.  `add`: to the partials of the chunks before.
__device__ void dot_chunk(const GSArgs& a, int64_t r0, int rows, const int4* ys, int Ky, int rb, bool add) {
  const int lane = threadIdx.x & 31, q = threadIdx.x >> 5;
  const int64_t n = a.n, h = a.h;
  const int j = a.j;
  int4 keep = make_int4(0, 0, 0, 0);
  int k = 0;
  for (int c = q; c <= j; c += kW) {
    const fxc* v = (const fxc*)a.V + (int64_t)c * n + r0;
    FxAcc s[7];
#pragma unroll
    for (int t = 0; t < 7; ++t) fx_zero(s[t]);
    int r = lane;
#pragma unroll 1
    for (; r + 32 < rows; r += 64) {
      const fxc a1 = v[r], a2 = v[h + r], b1 = v[r + 32], b2 = v[h + r + 32];
      dot_row(s, a1, a2, ys[r], ys[rows + r]);
      dot_row(s, b1, b2, ys[r + 32], ys[rows + r + 32]);
    }
    if (r < rows) dot_row(s, v[r], v[h + r], ys[r], ys[rows + r]);
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      const int4 p = fx_warp_sum(t == 0 ? s[0] : fx_diff(s[2 * t - 1], s[2 * t]));
      if (lane == 4 * k + t) keep = p;
    }
    if (++k == 8 || c + kW > j) {
      const int cl = c - kW * (k - 1 - (lane >> 2));       // this lane's column
      if ((lane >> 2) < k) {
        const double val = fx_value(keep, a.vexp[cl], Ky);
        double* out = a.part_dot + ((int64_t)cl * a.nblk + rb) * 4 + (lane & 3);
        *out = add ? *out + val : val;
      }
      k = 0;
    }
  }
}

// All chunks of one row block; returns this thread's share of ||y||^2 with SubAlpha.
template <bool SubAlpha>
__device__ double dot_block(const GSArgs& a, int64_t p0, int64_t p1, int4* ys, int* smax, double alpha, int rb) {
  double nrm = 0.0;
  for (int64_t r0 = p0; r0 < p1; r0 += kChunk) {
    const int rows = (int)min((int64_t)kChunk, p1 - r0);
    const int K = load_chunk<SubAlpha>(a, r0, rows, ys, smax, alpha, &nrm);
    dot_chunk(a, r0, rows, ys, K, rb, r0 > p0);
  }
  return nrm;
}

// ------------------------------------------------------------------ update
// The coefficients in shared memory, prepared once per launch (every block alike).  Column i contributes
// through its stored integers, so its coefficient is scaled by the column's 2^e_i.  A column is large when a
// component of c_v or c_w exceeds line 2^(e_min - e_i), line = 2^-30 ||y|| / ((j+1)(j+4)) and e_min the least
// exponent of the columns: then no scaled coefficient of a small column exceeds line 2^e_min.  Large columns
// (list) are applied with both limbs of both factors, on the scale 2^(KL - 1023) of the largest of them; the
// others with the leading limb of V (28 bits) and 22 bits of the coefficient on the scale 2^(KS - 1023) of the
// largest of theirs, at most 2 line 2^e_min, in one 64-bit sum: 2^28 2^22 times 4 (j+1) <= 2^12 terms stay below
// 2^63.  A component of a coefficient is off by less than 2^-22 (1 + 2^-5) line, which over the columns makes
// below 2^-50 / (j + 4) of ||y||; a component of V is off by less than 2^-28 of its column's scale, together below
// 2^-56 rho / (j + 4) of ||y||, rho = 2^e_min sqrt(2n), the peak of the flattest column over its rms (below 16 for
// a column of Gaussian entries).  Without the factor 2^(e_min - e_i) a small column with one entry near 1 set a
// scale on which the coefficients of flat columns kept up to 11 bits fewer (n = 4M).
// Rounding-size coefficients are about 2^-50 ||y||, far below the line for any j and for columns whose
// exponents are a few apart, so a step streams V once at 16 multiply-adds a row pair and column.
struct UpdFx {
  int4* sm;      // [m+1] small columns: c_v.re, c_v.im, c_w.re, c_w.im as integers (zero for a large one)
  int4* lg;      // [m+1][2] large columns: limbs of c_v (re, im), then of c_w
  int* list;     // [m+1] large columns, ascending
  int* misc;     // number of large columns, KS, KL
};
__host__ __device__ inline size_t upd_smem(int m) { return (size_t)(m + 1) * (3 * sizeof(int4) + sizeof(int)) + 16; }
__device__ __forceinline__ UpdFx upd_carve(unsigned char* p, int m) {
  UpdFx u;
  u.sm = (int4*)p;
  u.lg = u.sm + m + 1;
  u.list = (int*)(u.lg + 2 * (m + 1));
  u.misc = u.list + m + 1;
  return u;
}

// Classification and conversion of the coefficients; line: fx_line of the norm before the update.
__device__ __forceinline__ int coef_high(const coef4& c) {
  return max(max(fx_high(c.vr), fx_high(c.vi)), max(fx_high(c.wr), fx_high(c.wi)));
}
__device__ void classify(const GSArgs& a, int line, UpdFx u) {
  const int j = a.j;
  __syncthreads();                                    // the last pass's readers are done
  if (threadIdx.x < 3) u.misc[threadIdx.x] = 0;
  __syncthreads();
  const int emin = a.vmin[j];
  int fs = 0, fl = 0;
  for (int i = threadIdx.x; i <= j; i += kT) {
    const int m = coef_high(a.coef[i]), f = m >> 20;
    const bool large = fx_large(m, a.vexp[i] - emin, line);
    const int g = f ? max(f + a.vexp[i] - 1023, 1) : 0;     // exponent field of the scaled coefficient
    u.list[i] = large ? 1 : 0;
    if (large) fl = max(fl, g);
    else fs = max(fs, g);
  }
  fs = __reduce_max_sync(0xffffffffu, fs);
  fl = __reduce_max_sync(0xffffffffu, fl);
  if ((threadIdx.x & 31) == 0) {
    if (fs) atomicMax(u.misc + 1, fs);
    if (fl) atomicMax(u.misc + 2, fl);
  }
  __syncthreads();
  const int KS = u.misc[1] + 1, KL = u.misc[2] + 1;
  for (int i = threadIdx.x; i <= j; i += kT) {
    const coef4 c = a.coef[i];
    const int e = a.vexp[i] - 1023;
    if (u.list[i]) {
      const fx2 p = fx_limbs<true>(c.vr, KL - e), q = fx_limbs<true>(c.vi, KL - e);
      const fx2 r = fx_limbs<true>(c.wr, KL - e), t = fx_limbs<true>(c.wi, KL - e);
      u.lg[2 * i] = make_int4(p.h, p.l, q.h, q.l);
      u.lg[2 * i + 1] = make_int4(r.h, r.l, t.h, t.l);
      u.sm[i] = make_int4(0, 0, 0, 0);
    } else {
      u.sm[i] = make_int4((fx_limbs<true>(c.vr, KS - e).h + 32) >> 6, (fx_limbs<true>(c.vi, KS - e).h + 32) >> 6,
                          (fx_limbs<true>(c.wr, KS - e).h + 32) >> 6, (fx_limbs<true>(c.wi, KS - e).h + 32) >> 6);
    }
  }
  __syncthreads();
  if (threadIdx.x < 32) {                             // the large columns' list, in place of the flags
    int cnt = 0;
    for (int i0 = 0; i0 <= j; i0 += 32) {
      const int i = i0 + (int)threadIdx.x;
      const bool large = i <= j && u.list[i] != 0;
      const unsigned b = __ballot_sync(0xffffffffu, large);
      if (large) u.list[cnt + __popc(b & ((1u << threadIdx.x) - 1u))] = i;   // cnt + ... <= i
      __syncwarp();
      cnt += __popc(b);
    }
    if (threadIdx.x == 0) u.misc[0] = cnt;
  }
  __syncthreads();
}

// y1: v1 c_v - conj(v2) c_w;  y2: v2 c_v + conj(v1) c_w, by the leading limbs of v
__device__ __forceinline__ void small_row(long long* s, fxc v1, fxc v2, int4 c) {
  const int ax = (int)(v1.re >> 32), ay = (int)(v1.im >> 32), bx = (int)(v2.re >> 32), by = (int)(v2.im >> 32);
  const int ny = -c.y, nz = -c.z, nw = -c.w;
  fx_mad(s[0], ax, c.x); fx_mad(s[0], ay, ny); fx_mad(s[0], bx, nz); fx_mad(s[0], by, nw);
  fx_mad(s[1], ax, c.y); fx_mad(s[1], ay, c.x); fx_mad(s[1], bx, nw); fx_mad(s[1], by, c.z);
  fx_mad(s[2], bx, c.x); fx_mad(s[2], by, ny); fx_mad(s[2], ax, c.z); fx_mad(s[2], ay, c.w);
  fx_mad(s[3], bx, c.y); fx_mad(s[3], by, c.x); fx_mad(s[3], ax, c.w); fx_mad(s[3], ay, nz);
}
__device__ __forceinline__ void large_row(FxAcc* s, fxc v1, fxc v2, int4 cv, int4 cw) {
  const fx2 a = fx_round(v1.re), b = fx_round(v1.im), c = fx_round(v2.re), d = fx_round(v2.im);
  const fx2 p{cv.x, cv.y}, q{cv.z, cv.w}, r{cw.x, cw.y}, t{cw.z, cw.w};
  const fx2 nq = fx_neg(q), nr = fx_neg(r), nt = fx_neg(t);
  fx_mac(s[0], a, p); fx_mac(s[0], b, nq); fx_mac(s[0], c, nr); fx_mac(s[0], d, nt);
  fx_mac(s[1], a, q); fx_mac(s[1], b, p); fx_mac(s[1], c, nt); fx_mac(s[1], d, r);
  fx_mac(s[2], c, p); fx_mac(s[2], d, nq); fx_mac(s[2], a, r); fx_mac(s[2], b, t);
  fx_mac(s[3], c, q); fx_mac(s[3], d, p); fx_mac(s[3], a, t); fx_mac(s[3], b, nr);
}
struct RedFx {   // cross-warp sums of a tile that several warps share
  long long s[kW][4][32];
  double d[kW][4][32];
};
// dynamic shared memory of the cooperative step: limbs of y or the update's sums, then UpdFx
constexpr size_t kBuf = sizeof(RedFx) > 2 * kChunk * sizeof(int4) ? sizeof(RedFx) : 2 * kChunk * sizeof(int4);

// y -= V c_v + W c_w over rows [p0, p1), a lane a row pair; returns this thread's share of ||y||^2 and
// the largest |component| of y it wrote (its high word) in *ymax.  A block of few 32-row tiles lets
// `share` of its warps, a power of two, work on a tile, each with its columns; their sums meet in the
// first of them.  (Two row pairs a lane, for longer runs of a column a load, spilled and ran slower.)
__device__ double update_block(const GSArgs& a, int64_t p0, int64_t p1, UpdFx u, RedFx* red, int* ymax) {
  const int lane = threadIdx.x & 31, q = threadIdx.x >> 5;
  double2* y = (double2*)a.y;
  const int64_t n = a.n, h = a.h;
  const int j = a.j;
  const int tiles = (int)((p1 - p0 + 31) >> 5);
  int share = 1;
  while (share < kW && 2 * share * tiles <= kW) share *= 2;
  const int group = kW / share;                             // tiles at a time; the warps of a tile q, q + group, ...:
  const int tq = q % group, sub = q / group;                // its first warp, which works in FP64, on a quarter of its own
  const int nl = u.misc[0], KS = u.misc[1] + 1, KL = u.misc[2] + 1;
  double nrm = 0.0;
  int ym = 0;
  for (int t0 = 0; t0 < tiles; t0 += group) {
    const int64_t p = p0 + 32 * (int64_t)(t0 + tq) + lane;
    const bool ok = p < p1;
    long long s[4] = {0, 0, 0, 0};
    double d[4] = {0.0, 0.0, 0.0, 0.0};
    double2 y1 = make_double2(0.0, 0.0), y2 = y1;
    if (ok) {
      if (sub == 0) {
        y1 = y[p];
        y2 = y[h + p];
      }
      const fxc* v = (const fxc*)a.V + p;
      constexpr int U = 4;
      fxc a1[U], a2[U], b1[U], b2[U];
      auto fetch = [&](int i, fxc* v1, fxc* v2) {
#pragma unroll
        for (int t = 0; t < U; ++t)
          if (i + t * share <= j) {
            v1[t] = v[(int64_t)(i + t * share) * n];
            v2[t] = v[(int64_t)(i + t * share) * n + h];
          }
      };
      auto work = [&](int i, const fxc* v1, const fxc* v2) {
#pragma unroll
        for (int t = 0; t < U; ++t)
          if (i + t * share <= j) small_row(s, v1[t], v2[t], u.sm[i + t * share]);
      };
      fetch(sub, a1, a2);
      for (int i = sub; i <= j; i += 2 * U * share) {
        fetch(i + U * share, b1, b2);
        work(i, a1, a2);
        fetch(i + 2 * U * share, a1, a2);
        work(i + U * share, b1, b2);
      }
      for (int l0 = sub; l0 < nl; l0 += 16 * share) {       // at most 64 products a sum
        FxAcc f[4];
#pragma unroll
        for (int t = 0; t < 4; ++t) fx_zero(f[t]);
        for (int l = l0; l < min(nl, l0 + 16 * share); l += share) {
          const int k = u.list[l];
          large_row(f, v[(int64_t)k * n], v[(int64_t)k * n + h], u.lg[2 * k], u.lg[2 * k + 1]);
        }
#pragma unroll
        for (int t = 0; t < 4; ++t) {
          const double x = fx_lane_value(f[t], KL);
          d[t] = l0 == sub ? x : d[t] + x;
        }
      }
    }
    if (share > 1) {
      if (sub > 0)
#pragma unroll
        for (int t = 0; t < 4; ++t) {
          red->s[q][t][lane] = s[t];
          red->d[q][t][lane] = d[t];
        }
      __syncthreads();
      if (sub == 0)
        for (int g = 1; g < share; ++g)
#pragma unroll
          for (int t = 0; t < 4; ++t) {
            s[t] += red->s[q + g * group][t][lane];
            if (g < nl) d[t] += red->d[q + g * group][t][lane];
          }
      __syncthreads();
    }
    if (ok && sub == 0) {
#pragma unroll
      for (int t = 0; t < 4; ++t) d[t] += fx_to_double(s[t] >> 63, (unsigned long long)s[t], KS - 1023 - 50);
      y1.x -= d[0];
      y1.y -= d[1];
      y2.x -= d[2];
      y2.y -= d[3];
      y[p] = y1;
      y[h + p] = y2;
      nrm += cabs2(y1) + cabs2(y2);
      ym = max(ym, max(max(__double2hiint(y1.x) & 0x7fffffff, __double2hiint(y1.y) & 0x7fffffff),
                       max(__double2hiint(y2.x) & 0x7fffffff, __double2hiint(y2.y) & 0x7fffffff)));
    }
  }
  *ymax = ym;
  return nrm;
}

// Largest int over the block: of one a thread, or of cnt in memory.
__device__ __forceinline__ int block_imax(int v, int* smax) {
  v = __reduce_max_sync(0xffffffffu, v);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) smax[threadIdx.x >> 5] = v;
  __syncthreads();
#pragma unroll
  for (int w = 0; w < kW; ++w) v = max(v, smax[w]);
  return v;
}
__device__ __forceinline__ int block_imax(const int* src, int cnt, int* smax) {
  int v = 0;
  for (int b = threadIdx.x; b < cnt; b += kT) v = max(v, src[b]);
  return block_imax(v, smax);
}

// v_{j+1} = y inv over rows [p0, p1) into the basis and into x (FP64, the next product's input).  ymax:
// high word of the largest |component| of y, which gives the column's exponent.
__device__ void normalize_block(const GSArgs& a, int64_t p0, int64_t p1, double inv, int ymax) {
  const double2* y = (const double2*)a.y;
  fxc* v = (fxc*)a.V + (int64_t)(a.j + 1) * a.n;
  const int K = fx_field(__hiloint2double(ymax + 1, 0) * inv) + 1;
  if (p0 == 0 && threadIdx.x == 0) {
    a.vexp[a.j + 1] = K;
    a.vmin[a.j + 1] = min(a.vmin[a.j], K);
  }
  const int64_t rows = p1 - p0;
  for (int64_t e = threadIdx.x; e < 2 * rows; e += kT) {
    const int64_t i = p0 + (e < rows ? e : e - rows + a.h);
    const double2 t = y[i];
    const double2 w = make_double2(t.x * inv, t.y * inv);
    v[i] = fxc{fx_store(w.x, K), fx_store(w.y, K)};
    a.x[i] = w;
  }
}

// Sum of cnt doubles (src, stride) over the block in a fixed order; `then` runs on thread 0 with it and
// what it returns is every thread's result.  The partial sums of the warps are integer (fixed.cuh): with
// FP64 adds in every warp of every block the FP64 pipe made one such sum take 7,000 clocks at 384 blocks.
template <typename F>
__device__ __forceinline__ double block_dsum(const double* src, int stride, int cnt, double* sh, F then) {
  const int w = threadIdx.x >> 5;
  const bool live = 32 * w < cnt;
  const double s = live ? fx_warp_dsum(src, stride, threadIdx.x, cnt, kT) : 0.0;
  __syncthreads();
  if ((threadIdx.x & 31) == 0) sh[w] = s;
  __syncthreads();
  if (threadIdx.x < 32) {
    const int nw = min(kW, (cnt + 31) >> 5);
    double t = (int)threadIdx.x < nw ? sh[threadIdx.x] : 0.0;
    for (int o = 1; o < nw; o <<= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if (threadIdx.x == 0) sh[kW] = then(t);
  }
  __syncthreads();
  return sh[kW];
}
__device__ __forceinline__ double block_dsum(const double* src, int stride, int cnt, double* sh) {
  return block_dsum(src, stride, cnt, sh, [](double s) { return s; });
}
__device__ __forceinline__ double block_dnorm(const double* part, int cnt, double* sh) {
  return block_dsum(part, 1, cnt, sh, [](double s) { return sqrt(s); });
}

// Sum over the block of one double a thread; thread 0 gets it.  A warp of zeros costs no FP64 instruction.
__device__ __forceinline__ double block_total(double v, double* sh) {
  const int w = threadIdx.x >> 5;
  if (__any_sync(0xffffffffu, __double_as_longlong(v) != 0)) v = warp_sum(v);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) sh[w] = v;
  __syncthreads();
  double t = 0.0;
  if (threadIdx.x < 32) {
    t = (int)threadIdx.x < kW ? sh[threadIdx.x] : 0.0;
    for (int o = 1; o < kW; o <<= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
  }
  return t;
}

// The step's bookkeeping of alpha (t_{j,j} its real part);
// thread 0 of the lead block.  tmax: max |t| with alpha.
__device__ __forceinline__ double tmax_with(const GSArgs& a, double ar) {
  double tm = fmax(a.st->tmax, fabs(ar));
  if (a.j > 0) tm = fmax(tm, fabs(a.T[(int64_t)a.j * a.ldt + a.j - 1]));
  return tm;
}
__device__ void record_alpha(const GSArgs& a, double ar) {
  const int j = a.j;
  StepState* st = a.st;
  st->done = 0;
  st->tmax = tmax_with(a, ar);
  a.T[(int64_t)j * a.ldt + j] = ar;
  st->n_passes += 1;
  st->units_first += (double)(j + 1) * (double)a.h;
}

// ------------------------------------------------------------------ separate launches
__global__ void __launch_bounds__(kT, 1)
gsfx_first_kernel(GSArgs a, const double2* __restrict__ alpha_part, int n_alpha_part) {
  __shared__ double sh[32];
  __shared__ int smax[kW];
  __shared__ int4 ys[2 * kChunk];
  const double ar = block_dsum((const double*)alpha_part, 2, n_alpha_part, sh);
  if (blockIdx.x == 0) {
    const double ai = block_dsum((const double*)alpha_part + 1, 2, n_alpha_part, sh);
    if (threadIdx.x == 0) {
      record_alpha(a, ar);
      a.st->alpha_im = ai;
    }
  }
  const int64_t p0 = (int64_t)blockIdx.x * a.rows_per_block;
  const int64_t p1 = min(p0 + (int64_t)a.rows_per_block, a.h);
  const double nrm = block_total(dot_block<true>(a, p0, p1, ys, smax, ar, blockIdx.x), sh);
  if (threadIdx.x == 0) a.part_nrm[blockIdx.x] = nrm;
}

__global__ void __launch_bounds__(kT, 1) gsfx_dot_kernel(GSArgs a, int pass) {
  __shared__ double sh[32];
  __shared__ int smax[kW];
  __shared__ int4 ys[2 * kChunk];
  __shared__ int s_skip;
  StepState* st = a.st;
  if (threadIdx.x == 0) s_skip = st->done;
  __syncthreads();
  if (s_skip) return;
  const double nrm_prev = block_dnorm(a.part_nrm, a.nblk, sh);   // b1 after pass - 1
  const double ref = st->nrm[pass - 2];              // b0 before pass - 1
  const bool exits = kSqrt2 * nrm_prev > ref;
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    st->nrm[pass - 1] = nrm_prev;
    if (exits) {
      st->beta = nrm_prev;
      st->done = 1;
    } else {
      st->n_passes += 1;
      st->units_dot += (double)(a.j + 1) * (double)a.h;
    }
  }
  if (exits) return;
  const int64_t p0 = (int64_t)blockIdx.x * a.rows_per_block;
  const int64_t p1 = min(p0 + (int64_t)a.rows_per_block, a.h);
  dot_block<false>(a, p0, p1, ys, smax, 0.0, blockIdx.x);
}

__global__ void __launch_bounds__(kT, 1) gsfx_update_kernel(GSArgs a, int pass) {
  extern __shared__ __align__(32) unsigned char dyn[];
  __shared__ double sh[32];
  __shared__ int smax[kW];
  __shared__ int s_skip;
  if (threadIdx.x == 0) s_skip = a.st->done;
  __syncthreads();
  if (s_skip) return;
  const UpdFx u = upd_carve(dyn + kBuf, a.m);
  classify(a, fx_line(a.st->nrm[pass - 1], a.j), u);             // ||y|| before this update
  if (blockIdx.x == 0 && threadIdx.x == 0) a.st->units_update += (double)(a.j + 1) * (double)a.h;
  const int64_t p0 = (int64_t)blockIdx.x * a.rows_per_block;
  const int64_t p1 = min(p0 + (int64_t)a.rows_per_block, a.h);
  int ym;
  const double nrm = block_total(update_block(a, p0, p1, u, (RedFx*)dyn, &ym), sh);
  ym = block_imax(ym, smax);
  if (threadIdx.x == 0) {
    a.part_nrm[blockIdx.x] = nrm;
    a.part_max[blockIdx.x] = ym;
  }
}

// v_{j+1} = y / beta; t_{j+1,j} = beta; breakdown check.
__device__ __forceinline__ void record_beta(const GSArgs& a, double beta, bool brk) {
  const int j = a.j;
  a.T[(int64_t)(j + 1) * a.ldt + j] = beta;
  if (j + 1 < a.m) a.T[(int64_t)j * a.ldt + j + 1] = beta;
  if (brk) a.st->status = 5;
}

__global__ void __launch_bounds__(kT) gsfx_normalize_kernel(GSArgs a) {
  __shared__ double sh[32];
  __shared__ int smax[kW];
  const StepState* st = a.st;
  const int ym = block_imax(a.part_max, a.nblk, smax);
  double beta;
  if (st->done) {
    beta = st->beta;
  } else {  // the pass cap was reached: keep the norm after the last pass
    beta = block_dnorm(a.part_nrm, a.nblk, sh);
  }
  const bool brk = !(beta > 1e-14 * fmax(st->tmax, 1.0));
  const int64_t p0 = (int64_t)blockIdx.x * a.rows_per_block;
  const int64_t p1 = min(p0 + (int64_t)a.rows_per_block, a.h);
  normalize_block(a, p0, p1, brk ? 0.0 : 1.0 / beta, ym);
  if (blockIdx.x == 0 && threadIdx.x == 0) record_beta(a, beta, brk);
}

// ------------------------------------------------------------------ one cooperative launch per step
// The whole Gram-Schmidt part of one Lanczos step (alpha, y -= alpha v_j, every pass of dot, reduce and
// update with the sqrt(2) test, normalisation) in a single cooperative launch of one block per row block;
// the grid synchronises where the separate launches end one and start the next.  Every block computes the
// norms of the test from the same partials in the same order, so all take the same decision.  nrm2 holds
// two slots of nblk norm partials, alternating between passes.
// Cluster: the grid is one thread-block cluster, which synchronises in hardware (a grid-wide barrier takes
// about 3,000 clocks).
template <bool Cluster>
__global__ void __launch_bounds__(kT, 1)
gsfx_step_coop_kernel(GSArgs a, const double2* alpha_part, int n_alpha_part, int passes, double* nrm2) {
  namespace cg = cooperative_groups;
  auto sync_all = [] {
    if constexpr (Cluster) cg::this_cluster().sync();
    else cg::this_grid().sync();
  };
  __shared__ double sh[32];
  __shared__ int smax[kW];
  __shared__ double s_inv;
  __shared__ int s_exit;
  extern __shared__ __align__(32) unsigned char dyn[];
  int4* ys = (int4*)dyn;                             // during the dots
  RedFx* red = (RedFx*)dyn;                          // during the updates
  const UpdFx u = upd_carve(dyn + kBuf, a.m);
  const int j = a.j, nblk = a.nblk, rb = blockIdx.x;
  const int64_t h = a.h;
  const int64_t p0 = (int64_t)rb * a.rows_per_block;
  const int64_t p1 = min(p0 + (int64_t)a.rows_per_block, h);
  StepState* st = a.st;
  const bool lead = blockIdx.x == 0 && threadIdx.x == 0;
  dep_wait();
  dep_trigger();
  double tmax = 0.0;                                 // thread 0 of every block
  if (threadIdx.x == 0) tmax = a.st->tmax;
  const double ar = block_dsum((const double*)alpha_part, 2, n_alpha_part, sh);   // every block, the same order
  if (threadIdx.x == 0) {
    tmax = fmax(tmax, fabs(ar));
    if (j > 0) tmax = fmax(tmax, fabs(a.T[(int64_t)j * a.ldt + j - 1]));
  }
  {
    const double nb = block_total(dot_block<true>(a, p0, p1, ys, smax, ar, rb), sh);
    if (threadIdx.x == 0) nrm2[rb] = nb;
  }
  double bref = 0.0;
  int ymax = 0;
  for (int pass = 1;; ++pass) {
    sync_all();                                           // dot partials and norm partials complete
    if (pass == 1) {
      if (lead) record_alpha(a, ar);                       // after every block has read st->tmax
      bref = block_dnorm(nrm2, nblk, sh);                  // b0
      if (lead) st->nrm[0] = bref;
    }
    const int comps = 4 * (j + 1);
    if (comps <= nblk) {                                   // one component of a coefficient a block, or a warp
      if (rb < comps) {
        const double s = block_dsum(a.part_dot + (int64_t)(rb >> 2) * nblk * 4 + (rb & 3), 4, nblk, sh);
        if (threadIdx.x == 0) ((double*)a.coef)[rb] = (a.no_w && (rb & 2)) ? 0.0 : s;
      }
    } else {
      for (int c = rb + nblk * (int)(threadIdx.x >> 5); c < comps; c += nblk * kW) {
        const double s = fx_warp_dsum(a.part_dot + (int64_t)(c >> 2) * nblk * 4 + (c & 3), 4, threadIdx.x & 31, nblk, 32);
        if ((threadIdx.x & 31) == 0) ((double*)a.coef)[c] = (a.no_w && (c & 2)) ? 0.0 : s;
      }
    }
    sync_all();                                           // coefficients complete
    classify(a, fx_line(bref, j), u);
    double* slot = nrm2 + (size_t)(pass & 1) * nblk;
    int* mslot = a.part_max + (size_t)(pass & 1) * nblk;
    {
      int ym;
      const double nb = block_total(update_block(a, p0, p1, u, red, &ym), sh);
      ym = block_imax(ym, smax);
      if (threadIdx.x == 0) {
        slot[rb] = nb;
        mslot[rb] = ym;
      }
    }
    if (lead) st->units_update += (double)(j + 1) * (double)h;
    sync_all();                                           // updated y and its norm partials complete
    const double b1 = block_dsum(slot, 1, nblk, sh, [&](double s) {
      const double b = sqrt(s);
      const bool exits = kSqrt2 * b > bref || pass >= passes;   // the sqrt(2) test, or the pass cap
      s_exit = exits;
      if (exits) {   // normalise: breakdown below 1e-14 max(max|t|, 1)
        const bool brk = !(b > 1e-14 * fmax(tmax, 1.0));
        s_inv = brk ? 0.0 : 1.0 / b;
        if (lead) {
          st->beta = b;
          st->done = 1;
          record_beta(a, b, brk);
        }
      } else if (lead) {
        st->n_passes += 1;
        st->units_dot += (double)(j + 1) * (double)h;
      }
      if (lead && pass < 8) st->nrm[pass] = b;
      return b;
    });
    if (s_exit) {
      ymax = block_imax(mslot, nblk, smax);
      break;
    }
    bref = b1;
    dot_block<false>(a, p0, p1, ys, smax, 0.0, rb);
  }
  normalize_block(a, p0, p1, s_inv, ymax);                 // v_{j+1} = y / beta
  if (rb == nblk - 1) {                                    // Im(v_j^H A v_j), a diagnostic
    const double ai = block_dsum((const double*)alpha_part + 1, 2, n_alpha_part, sh);
    if (threadIdx.x == 0) st->alpha_im = ai;
  }
}

size_t fx_smem(int m) { return kBuf + upd_smem(m); }

// ------------------------------------------------------------------ columns in and out of the basis
// kmax[c] = largest exponent field of the FP64 column c (perm[c] if given) + 1, for a zeroed kmax
__global__ void col_field_kernel(const double2* X, int64_t n, const int* perm, int* kmax) {
  const int c = blockIdx.y;
  const double2* x = X + (int64_t)(perm ? perm[c] : c) * n;
  int ex = 0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const double2 v = x[i];
    ex = max(ex, max(fx_field(v.x), fx_field(v.y)));
  }
  ex = __reduce_max_sync(0xffffffffu, ex);
  if ((threadIdx.x & 31) == 0) atomicMax(kmax + c, ex + 1);
}
// V[:, c] = X[:, perm[c]] (perm null: c) with the exponents kmax for c < k; V[:, k] = V[:, m] if k < m
// (the restart's shrink of Algorithm 1).
__global__ void store_cols_kernel(fxc* V, const double2* X, int64_t n, const int* perm, int k, int m, int* vexp,
                                  int* vmin, const int* kmax) {
  const int c = blockIdx.y;
  fxc* dst = V + (int64_t)c * n;
  const int64_t i0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, di = (int64_t)gridDim.x * blockDim.x;
  if (i0 == 0) {
    int e = c < k ? kmax[c] : vexp[m];
    for (int i = 0; i < min(c, k); ++i) e = min(e, kmax[i]);
    vmin[c] = e;
  }
  if (c < k) {
    const double2* src = X + (int64_t)(perm ? perm[c] : c) * n;
    const int K = kmax[c];
    if (i0 == 0) vexp[c] = K;
    for (int64_t i = i0; i < n; i += di) {
      const double2 v = src[i];
      dst[i] = fxc{fx_store(v.x, K), fx_store(v.y, K)};
    }
  } else {
    const fxc* src = V + (int64_t)m * n;
    if (i0 == 0) vexp[c] = vexp[m];
    for (int64_t i = i0; i < n; i += di) dst[i] = src[i];
  }
}
// Column V in FP64.
__global__ void load_col_kernel(const fxc* V, const int* vexp, int64_t n, double2* x) {
  const int K = *vexp;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const fxc v = V[i];
    x[i] = make_double2(fx_load(v.re, K), fx_load(v.im, K));
  }
}
// out[:, c] = X[:, perm[order[c]]] and, with partners, out[:, nev + c] = J conj(...) = [-x2^*; x1^*].
__global__ void gather_pairs_kernel(const double2* X, const int* perm, int64_t n, const int* order, int nev, int partners,
                                    double2* out) {
  const int c = blockIdx.y;
  const int64_t h = n / 2;
  const double2* src = X + (int64_t)perm[order[c]] * n;
  double2* dst = out + (int64_t)c * n;
  double2* dstp = out + (int64_t)(nev + c) * n;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < h; i += (int64_t)gridDim.x * blockDim.x) {
    const double2 x1 = src[i], x2 = src[h + i];
    dst[i] = x1;
    dst[h + i] = x2;
    if (partners) {
      dstp[i] = make_double2(-x2.x, x2.y);
      dstp[h + i] = make_double2(x1.x, -x1.y);
    }
  }
}

inline unsigned col_grid(int64_t n) {
  const int64_t g = (n + 1023) / 1024;
  return (unsigned)(g > 304 ? 304 : g);
}

}  // namespace

cudaError_t launch_store_cols(void* V, const void* X, int64_t n, const int* perm, int k, int m, int* vexp, int* vmin,
                              int* kmax, cudaStream_t s) {
  if (k > 0) {   // k = 0: a restart that keeps v_{m+1} alone
    cudaError_t e = cudaMemsetAsync(kmax, 0, (size_t)k * sizeof(int), s);
    if (e != cudaSuccess) return e;
    col_field_kernel<<<dim3(col_grid(n), k), 256, 0, s>>>((const double2*)X, n, perm, kmax);
  }
  store_cols_kernel<<<dim3(col_grid(n), k < m ? k + 1 : k), 256, 0, s>>>((fxc*)V, (const double2*)X, n, perm, k, m, vexp,
                                                                        vmin, kmax);
  return cudaGetLastError();
}

cudaError_t launch_field(const void* X, int64_t n, int* kmax, cudaStream_t s) {
  cudaError_t e = cudaMemsetAsync(kmax, 0, sizeof(int), s);
  if (e != cudaSuccess) return e;
  col_field_kernel<<<dim3(col_grid(n)), 256, 0, s>>>((const double2*)X, n, nullptr, kmax);
  return cudaGetLastError();
}

cudaError_t launch_load_col(const void* V, const int* vexp, int64_t n, int c, double2* x, cudaStream_t s) {
  load_col_kernel<<<col_grid(n) * 4, 256, 0, s>>>((const fxc*)V + (int64_t)c * n, vexp + c, n, x);
  return cudaGetLastError();
}

cudaError_t launch_gather_pairs(const void* X, const int* perm, int64_t n, const int* order, int nev, int partners,
                                void* out, cudaStream_t s) {
  gather_pairs_kernel<<<dim3(col_grid(n / 2), nev), 256, 0, s>>>((const double2*)X, perm, n, order, nev, partners,
                                                                (double2*)out);
  return cudaGetLastError();
}

template <>
cudaError_t launch_gs_first<double>(const GSArgs& a, const double2* alpha_part, int n_alpha_part, cudaStream_t s) {
  gsfx_first_kernel<<<a.nblk, kT, 0, s>>>(a, alpha_part, n_alpha_part);
  return cudaGetLastError();
}
template <>
cudaError_t launch_gs_update<double>(const GSArgs& a, int pass, cudaStream_t s) {
  const size_t sm = fx_smem(a.m);
  cudaError_t e = allow_dyn_smem((const void*)gsfx_update_kernel, sm);
  if (e != cudaSuccess) return e;
  gsfx_update_kernel<<<a.nblk, kT, sm, s>>>(a, pass);
  return cudaGetLastError();
}
template <>
cudaError_t launch_gs_dot<double>(const GSArgs& a, int pass, cudaStream_t s) {
  gsfx_dot_kernel<<<a.nblk, kT, 0, s>>>(a, pass);
  return cudaGetLastError();
}
template <>
cudaError_t launch_gs_normalize<double>(const GSArgs& a, cudaStream_t s) {
  gsfx_normalize_kernel<<<a.nblk, kT, 0, s>>>(a);
  return cudaGetLastError();
}
template <>
cudaError_t gs_coop_occupancy<double>(int m, int* per_sm) {
  int dev = 0, coop = 0, per = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev)) != cudaSuccess) return e;
  const size_t sm = fx_smem(m);
  if ((e = allow_dyn_smem((const void*)gsfx_step_coop_kernel<false>, sm)) != cudaSuccess) return e;
  if ((e = allow_dyn_smem((const void*)gsfx_step_coop_kernel<true>, sm)) != cudaSuccess) return e;
  if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, gsfx_step_coop_kernel<false>, kT, sm)) != cudaSuccess)
    return e;
  *per_sm = coop ? per : 0;
  return cudaSuccess;
}
template <>
cudaError_t launch_gs_step_coop<double>(const GSArgs& a, const double2* alpha_part, int n_alpha_part, int passes,
                                        double* nrm2, int grid, cudaStream_t s) {
  if (grid != a.nblk) return cudaErrorInvalidValue;   // one row block per CTA
  GSArgs aa = a;
  const double2* ap = alpha_part;
  int na = n_alpha_part, ps = passes;
  double* nr = nrm2;
  void* args[] = {&aa, &ap, &na, &ps, &nr};
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(kT);
  cfg.dynamicSmemBytes = fx_smem(a.m);
  cfg.stream = s;
  cudaLaunchAttribute at[2] = {};
  cfg.attrs = at;
  cfg.numAttrs = 1;
  if (grid <= kClusterMax) {   // the portable cluster size; one cluster, set up while the product ends
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = grid;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.numAttrs = 2;
    return cudaLaunchKernelExC(&cfg, (const void*)gsfx_step_coop_kernel<true>, args);
  }
  at[0].id = cudaLaunchAttributeCooperative;
  at[0].val.cooperative = 1;
  return cudaLaunchKernelExC(&cfg, (const void*)gsfx_step_coop_kernel<false>, args);
}

}  // namespace jtr
