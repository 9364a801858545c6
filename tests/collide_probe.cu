// Kernels of test_gpu_collide_probe.py: the helpers of lbm_collide.cuh against
// CUDA's own results and against the scalar collisions, cell by cell.
#include "lbm_collide.cuh"

using namespace lbm;

namespace {

template <typename F, typename G>
__device__ void count_range(unsigned lo, unsigned hi, unsigned long long *n, F f, G g) {
  unsigned long long bad = 0;
  for (unsigned long long b = lo + blockIdx.x * blockDim.x + threadIdx.x; b < hi;
       b += (unsigned long long)gridDim.x * blockDim.x) {
    const float x = __uint_as_float((unsigned)b);
    bad += __float_as_uint(f(x)) != __float_as_uint(g(x));
  }
  if (bad) atomicAdd(n, bad);
}
__global__ void k_rcp(unsigned lo, unsigned hi, unsigned long long *n) {
  count_range(lo, hi, n, [](float x) { return rcp_newton(x); },
              [](float x) { return __frcp_rn(x); });
}
__global__ void k_sqrt(unsigned lo, unsigned hi, unsigned long long *n) {
  count_range(lo, hi, n, [](float x) { return sqrt_newton(x); },
              [](float x) { return __fsqrt_rn(x); });
}

// cells: [2 n][9] deviations from rho0 t; one thread per pair.  out_pair the
// packed form, out_one the scalar one, taken[i] whether the packed form took the
// pair (it leaves pairs whose root needs iterations).
template <bool FORCED, bool ELBM>
__global__ void k_pairs(const float *cells, int n, float rho0, float tau, float fx, float fy,
                        float alpha, float *out_pair, float *out_one, int *taken) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  float a[kQ], b[kQ];
  f32x2 g[kQ];
  for (int l = 0; l < kQ; ++l) {
    a[l] = cells[(size_t)(2 * i) * kQ + l];
    b[l] = cells[(size_t)(2 * i + 1) * kQ + l];
    g[l] = pack2(a[l], b[l]);
  }
  bool ok = true;
  if (ELBM)
    ok = collide2_elbm<FORCED>(g, rho0, 2.0f * tau, both2(fx), both2(fy), alpha);
  else
    collide2_f32<FORCED>(g, rho0, 1.0f / tau, both2(fx), both2(fy), alpha);
  if (ELBM) {
    collide_elbm_call(a, rho0, tau, fx, fy, alpha);
    collide_elbm_call(b, rho0, tau, fx, fy, alpha);
  } else {
    collide_f32(a, rho0, 1.0f / tau, fx, fy, alpha);
    collide_f32(b, rho0, 1.0f / tau, fx, fy, alpha);
  }
  taken[i] = ok;
  for (int l = 0; l < kQ; ++l) {
    float pa, pb;
    unpack2(g[l], pa, pb);
    out_pair[(size_t)(2 * i) * kQ + l] = pa;
    out_pair[(size_t)(2 * i + 1) * kQ + l] = pb;
    out_one[(size_t)(2 * i) * kQ + l] = a[l];
    out_one[(size_t)(2 * i + 1) * kQ + l] = b[l];
  }
}

}  // namespace

extern "C" {

// Floats of [lo, hi) (as bits) whose reciprocal (what = 0) or square root (1)
// differs from CUDA's correctly rounded one; -1 on a CUDA error.
long long probe_count(int what, unsigned lo, unsigned hi) {
  unsigned long long *d = nullptr, n = 0;
  if (cudaMalloc(&d, sizeof n) != cudaSuccess) return -1;
  cudaMemset(d, 0, sizeof n);
  if (what == 0)
    k_rcp<<<1024, 256>>>(lo, hi, d);
  else
    k_sqrt<<<1024, 256>>>(lo, hi, d);
  const cudaError_t e = cudaMemcpy(&n, d, sizeof n, cudaMemcpyDeviceToHost);
  cudaFree(d);
  return e == cudaSuccess ? (long long)n : -1;
}

int probe_pairs(int elbm, int forced, const float *cells, int n, float rho0, float tau, float fx,
                float fy, float alpha, float *out_pair, float *out_one, int *taken) {
  const int g = (n + 127) / 128;
  if (elbm && forced)
    k_pairs<true, true><<<g, 128>>>(cells, n, rho0, tau, fx, fy, alpha, out_pair, out_one, taken);
  else if (elbm)
    k_pairs<false, true><<<g, 128>>>(cells, n, rho0, tau, fx, fy, alpha, out_pair, out_one, taken);
  else if (forced)
    k_pairs<true, false><<<g, 128>>>(cells, n, rho0, tau, fx, fy, alpha, out_pair, out_one, taken);
  else
    k_pairs<false, false><<<g, 128>>>(cells, n, rho0, tau, fx, fy, alpha, out_pair, out_one, taken);
  return (int)cudaDeviceSynchronize();
}

}  // extern "C"
