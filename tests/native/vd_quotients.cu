// The library's quotients from shared reciprocals beside the divisions they
// stand for, on arrays: q = a / b.
#include "vd_device.cuh"
#include "vd_div64.cuh"

__global__ void k_div64(const double* a, const double* b, int n, double* fast, double* div) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  fast[i] = ka_div(a[i], b[i], ka_rcp(b[i]));
  div[i] = a[i] / b[i];
}

__global__ void k_div2(const float* a, const float* b, int n, float* fast, float* div) {
  const int i = 2 * (blockIdx.x * blockDim.x + threadIdx.x);
  if (i + 1 >= n) return;
  const vd_f2 q = vd_div2(vd_pack(a[i], a[i + 1]), vd_pack(-b[i], -b[i + 1]),
                          vd_pack(__frcp_rn(b[i]), __frcp_rn(b[i + 1])));
  fast[i] = vd_lo(q);
  fast[i + 1] = vd_hi(q);
  div[i] = a[i] / b[i];
  div[i + 1] = a[i + 1] / b[i + 1];
}

extern "C" int q_div64(const double* a, const double* b, int n, double* fast, double* div) {
  k_div64<<<(n + 255) / 256, 256>>>(a, b, n, fast, div);
  return cudaDeviceSynchronize();
}
extern "C" int q_div2(const float* a, const float* b, int n, float* fast, float* div) {
  k_div2<<<(n / 2 + 255) / 256, 256>>>(a, b, n, fast, div);
  return cudaDeviceSynchronize();
}
