// Device arithmetic of the kernels on given operands, one call per function: out receives the results
// of n operand sets.  The net update of a cell is built with the FP32 units' flags (see build.py).
#include <cuda_runtime.h>

#include "fx_stage.cuh"
#include "fx_ye.cuh"

namespace {

template <int D> __global__ void net_kernel(const float* in, float* out, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  // per set: upper and lower flux of D directions, then the D factors; the pair's halves hold the set and
  // its mirror image
  fx::F2 up[3], lo[3], h[3], mh[3];
  for (int d = 0; d < 3; ++d) {
    const bool has = d < D;
    const float u = has ? in[(2 * d) * n + i] : 0.0f, l = has ? in[(2 * d + 1) * n + i] : 0.0f;
    const float x = has ? in[(2 * D + d) * n + i] : 0.0f;
    up[d] = fx::F2(u, -u);
    lo[d] = fx::F2(l, -l);
    h[d] = fx::F2(x);
    mh[d] = fx::F2(-x);
  }
  const int m = D - 1;
  const fx::F2 r = fx::net_update<D>(up[0], lo[0], up[1], lo[1], up[m], lo[m], h, mh);
  out[i] = r.x;
  out[n + i] = r.y;
}

// sums of n terms by one thread each: of x, of x - y, of x y with x = (float)x + (float)(x - (float)x)
__global__ void pair_kernel(const double* x, const float* y, double* out, int n, int m) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= m) return;
  fx::FPair a = {0.0f, 0.0f}, d = a, p = a;
  for (int k = 0; k < n; ++k) {
    const double xk = x[k * m + i];
    const float xh = (float)xk, xl = (float)(xk - (double)xh), yk = y[k * m + i];
    fx::acc(a, xh);
    fx::acc_diff(d, xh, yk);
    fx::acc_mul(p, xh, xl, yk);
  }
  out[i] = fx::val(a);
  out[m + i] = fx::val(d);
  out[2 * m + i] = fx::val(p);
}

}  // namespace

// m sums of n terms each (device arrays [n][m]; out [3][m])
extern "C" int arith_pairs(const double* x, const float* y, double* out, int n, int m) {
  pair_kernel<<<(m + 127) / 128, 128>>>(x, y, out, n, m);
  return (int)cudaDeviceSynchronize();
}

// in: (3 D) x n floats, out: 2 x n floats (device).  Returns the CUDA error.
extern "C" int arith_net(int D, const float* in, float* out, int n) {
  const int nb = (n + 127) / 128;
  if (D == 1) net_kernel<1><<<nb, 128>>>(in, out, n);
  else if (D == 2) net_kernel<2><<<nb, 128>>>(in, out, n);
  else net_kernel<3><<<nb, 128>>>(in, out, n);
  return (int)cudaDeviceSynchronize();
}
