// Device arithmetic of the kernels on given operands, one call per function: out receives the results
// of n operand sets.  The net update of a cell is built with the FP32 units' flags (see build.py).
#include <cuda_runtime.h>

#include <cstring>
#include <vector>

#include "fx_planck.h"
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

// out = f(x) by the FP64 function of the given number (in the order of the test's list)
__global__ void fp64_kernel(int f, const double* x, double* out, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double v = x[i];
  out[i] = f == 0   ? fx::rcp64(v)
           : f == 1 ? fx::rcp_pos(v)
           : f == 2 ? fx::rcp_any(v)
           : f == 3 ? fx::rcp_fast(v)
           : f == 4 ? fx::rcp_ge1(v)
           : f == 5 ? fx::sqrt64(v)
           : f == 6 ? fx::sqrt_any(v)
                    : fx::rsqrt64(v);
}
__global__ void hpow_kernel(const double* x, const int* h, double* out, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) out[i] = fx::hpow(x[i], h[i]);
}
// Q, w and whether Q is the upper integral, at x = x16 / 16
__global__ void edge_kernel(const double* x16, const double* tab, const fx::PlanckCoef pc, double* out, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const fx::PlanckEdge<double> e = fx::planck_edge_tab(x16[i], tab, pc);
  out[i] = e.Q;
  out[n + i] = e.w;
  out[2 * n + i] = e.upper ? 1.0 : 0.0;
}
// B_g(T) and dB_g/dT of every group, by pairs, with a_N = 1: out [2][G][n]
__global__ void band_kernel(const fx::PlanckTable tab, const float* edge, const float* T, float* out, int G, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const fx::PlanckAt p = fx::planck_at(tab, 1.0f, T[i]);
  for (int pr = 0; pr < (G + 1) / 2; ++pr) {
    fx::F2 B, dB;
    fx::planck_pair(tab, p, pr, G, edge, B, dB);
    out[(2 * pr) * n + i] = B.x;
    out[(G + 2 * pr) * n + i] = dB.x;
    if (2 * pr + 1 < G) {
      out[(2 * pr + 1) * n + i] = B.y;
      out[(G + 2 * pr + 1) * n + i] = dB.y;
    }
  }
}

}  // namespace

extern "C" int arith_fp64(int f, const double* x, double* out, int n) {
  fp64_kernel<<<(n + 127) / 128, 128>>>(f, x, out, n);
  return (int)cudaDeviceSynchronize();
}
extern "C" int arith_hpow(const double* x, const int* h, double* out, int n) {
  hpow_kernel<<<(n + 127) / 128, 128>>>(x, h, out, n);
  return (int)cudaDeviceSynchronize();
}
extern "C" int arith_planck_edge(const double* x16, double* out, int n) {
  const std::vector<double>& t = fx::planck_edge_table();
  fx::PlanckCoef pc{};  // (the table is left for the exponential series only)
  for (int k = 1; k <= fx::NPLANCK_UP; ++k) pc.rn[k - 1] = 1.0 / k;
  double* d = nullptr;
  cudaError_t e = cudaMalloc(&d, t.size() * sizeof(double));
  if (e == cudaSuccess) e = cudaMemcpy(d, t.data(), t.size() * sizeof(double), cudaMemcpyHostToDevice);
  if (e == cudaSuccess) {
    edge_kernel<<<(n + 127) / 128, 128>>>(x16, d, pc, out, n);
    e = cudaDeviceSynchronize();
  }
  cudaFree(d);
  return (int)e;
}
// nodes: the host table [G][nu][4]; edge: G + 1 band edges (host); T, out on the device
extern "C" int arith_planck_bands(const float* nodes, int G, int nu, float u0, int node_major, const float* edge, const float* T,
                                  float* out, int n) {
  std::vector<float4> host((size_t)G * nu);
  std::memcpy(host.data(), nodes, host.size() * sizeof(float4));
  const std::vector<float4> t = fx::planck_device_table(host, G, nu, node_major != 0);
  float4* d = nullptr;
  float* ed = nullptr;
  cudaError_t e = cudaMalloc(&d, t.size() * sizeof(float4));
  if (e == cudaSuccess) e = cudaMalloc(&ed, (G + 1) * sizeof(float));
  if (e == cudaSuccess) e = cudaMemcpy(d, t.data(), t.size() * sizeof(float4), cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemcpy(ed, edge, (G + 1) * sizeof(float), cudaMemcpyHostToDevice);
  if (e == cudaSuccess) {
    fx::PlanckTable pt{};
    pt.tab = d;
    pt.nu = nu;
    pt.u0 = u0;
    pt.si = node_major ? (G + 1) / 2 : 1;
    pt.sg = node_major ? 1 : nu;
    band_kernel<<<(n + 127) / 128, 128>>>(pt, ed, T, out, G, n);
    e = cudaDeviceSynchronize();
  }
  cudaFree(d);
  cudaFree(ed);
  return (int)e;
}

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
