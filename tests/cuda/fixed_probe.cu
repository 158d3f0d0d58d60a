// fixed_probe.cu -- entry points for tests/test_gpu_fixed_helpers.py: the device helpers of fixed.cuh and one
// Gram-Schmidt step of gsfx.cu on columns that the test chooses.
#include "../../paper_2001_07428_gb300/csrc/gsfx.cu"

namespace jtr {

namespace {

__global__ void limbs_kernel(const double* x, int count, int K, int2* out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= count) return;
  const fx2 v = fx_limbs<true>(x[i], K);
  out[i] = make_int2(v.h, v.l);
}
__global__ void store_kernel(const double* x, int count, int K, long long* F, int2* rounded, double* back) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= count) return;
  F[i] = fx_store(x[i], K);
  const fx2 r = fx_round(F[i]);
  rounded[i] = make_int2(r.h, r.l);
  back[i] = fx_load(F[i], K);
}
// one warp: out[0] the sum of all cnt doubles, out[1] that of one double a lane
__global__ void sum_kernel(const double* x, int cnt, double* out) {
  const double a = fx_warp_dsum(x, 1, threadIdx.x, cnt, 32);
  const double b = fx_warp_total((int)threadIdx.x < cnt ? x[threadIdx.x] : 0.0);
  if (threadIdx.x == 0) {
    out[0] = a;
    out[1] = b;
  }
}

}  // namespace

extern "C" int probe_limbs(const double* x, int count, int K, int* out) {
  limbs_kernel<<<(count + 127) / 128, 128>>>(x, count, K, (int2*)out);
  return (int)cudaDeviceSynchronize();
}
extern "C" int probe_store(const double* x, int count, int K, long long* F, int* rounded, double* back) {
  store_kernel<<<(count + 127) / 128, 128>>>(x, count, K, F, (int2*)rounded, back);
  return (int)cudaDeviceSynchronize();
}
extern "C" int probe_sum(const double* x, int cnt, double* out) {
  sum_kernel<<<1, 32>>>(x, cnt, out);
  return (int)cudaDeviceSynchronize();
}

// One pass of the step against the cols columns of X (n x cols, FP64) in row blocks of rows_per_block row
// pairs: y (n) is orthogonalised in place, coef (4 doubles a column) receives c_v and c_w.
extern "C" int probe_step(const double* X, long long n, int cols, int rows_per_block, double* y, double* coef) {
  const int m = cols;
  const long long h = n / 2;
  const int nblk = (int)((h + rows_per_block - 1) / rows_per_block);
  char* base = nullptr;
  size_t used = 0;
  auto take = [&](size_t bytes) {
    const size_t at = used;
    used += (bytes + 255) / 256 * 256;
    return at;
  };
  const size_t oV = take((size_t)n * (m + 1) * sizeof(fxc)), ox = take((size_t)n * sizeof(double2));
  const size_t oT = take((size_t)(m + 1) * (m + 1) * sizeof(double)), oD = take((size_t)(m + 1) * nblk * sizeof(coef4));
  const size_t oN = take((size_t)2 * nblk * sizeof(double)), oM = take((size_t)2 * nblk * sizeof(int));
  const size_t oE = take((size_t)(m + 1) * sizeof(int)), oW = take((size_t)(m + 1) * sizeof(int)), oK = take((size_t)(m + 1) * sizeof(int));
  const size_t oS = take(sizeof(StepState)), oA = take(sizeof(double2));
  cudaError_t e = cudaMalloc((void**)&base, used);
  if (e != cudaSuccess) return (int)e;
  e = cudaMemset(base, 0, used);
  GSArgs a{};
  a.V = base + oV;
  a.n = n;
  a.h = h;
  a.j = cols - 1;
  a.y = y;
  a.part_dot = (double*)(base + oD);
  a.part_nrm = (double*)(base + oN);
  a.coef = (coef4*)coef;
  a.st = (StepState*)(base + oS);
  a.T = (double*)(base + oT);
  a.ldt = m + 1;
  a.m = m;
  a.nblk = nblk;
  a.rows_per_block = rows_per_block;
  a.vexp = (int*)(base + oE);
  a.vmin = (int*)(base + oW);
  a.part_max = (int*)(base + oM);
  a.x = (double2*)(base + ox);
  int per = 0;
  if (e == cudaSuccess) e = gs_coop_occupancy<double>(m, &per);
  if (e == cudaSuccess && (per < 1 || nblk > 152 * per)) e = cudaErrorInvalidValue;
  if (e == cudaSuccess) e = launch_store_cols((void*)a.V, X, n, nullptr, cols, cols, a.vexp, a.vmin, (int*)(base + oK), 0);
  if (e == cudaSuccess) e = launch_gs_step_coop<double>(a, (const double2*)(base + oA), 1, 1, a.part_nrm, nblk, 0);
  const cudaError_t s = cudaDeviceSynchronize();
  cudaFree(base);
  return (int)(e != cudaSuccess ? e : s);
}

}  // namespace jtr
