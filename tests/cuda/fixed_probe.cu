// fixed_probe.cu -- entry points for tests/test_gpu_fixed_helpers.py: the device helpers of fixed.cuh.
#include "../../paper_2001_07428_gb300/csrc/fixed.cuh"

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

}  // namespace jtr
