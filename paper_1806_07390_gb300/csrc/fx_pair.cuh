// Two FP32 values processed together: the two groups a lane owns in the stage kernel of the FP32
// forms.  Additions, subtractions, multiplications and fused multiply-adds use the packed FP32
// instructions of sm_100 and later (add/sub/mul/fma .f32x2: one instruction for both values,
// each rounded exactly as the scalar instruction would round it, denormals flushed as in the
// FP32 translation units).  Comparisons, selects, minima, reciprocals and square roots act on the
// two values one by one.
#pragma once
#include <cuda_runtime.h>

namespace fx {

struct alignas(8) F2 {
  float x, y;
  F2() = default;
  __host__ __device__ __forceinline__ F2(float a, float b) : x(a), y(b) {}
  __host__ __device__ __forceinline__ explicit F2(float a) : x(a), y(a) {}
};

// x as a lane value (both halves of a pair)
__host__ __device__ __forceinline__ F2 lane_value(float x, F2) { return F2(x); }
__host__ __device__ __forceinline__ double lane_value(double x, double) { return x; }

__device__ __forceinline__ unsigned long long f2_pack(F2 a) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a.x), "f"(a.y));
  return r;
}
__device__ __forceinline__ F2 f2_unpack(unsigned long long r) {
  F2 a;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a.x), "=f"(a.y) : "l"(r));
  return a;
}
__device__ __forceinline__ F2 operator+(F2 a, F2 b) {
  unsigned long long r;
  asm("add.rn.ftz.f32x2 %0, %1, %2;" : "=l"(r) : "l"(f2_pack(a)), "l"(f2_pack(b)));
  return f2_unpack(r);
}
__device__ __forceinline__ F2 operator-(F2 a, F2 b) {
  unsigned long long r;
  asm("sub.rn.ftz.f32x2 %0, %1, %2;" : "=l"(r) : "l"(f2_pack(a)), "l"(f2_pack(b)));
  return f2_unpack(r);
}
__device__ __forceinline__ F2 operator*(F2 a, F2 b) {
  unsigned long long r;
  asm("mul.rn.ftz.f32x2 %0, %1, %2;" : "=l"(r) : "l"(f2_pack(a)), "l"(f2_pack(b)));
  return f2_unpack(r);
}
__device__ __forceinline__ F2 operator-(F2 a) { return F2(-a.x, -a.y); }
__device__ __forceinline__ F2 operator+(F2 a, float b) { return a + F2(b); }
__device__ __forceinline__ F2 operator+(float a, F2 b) { return F2(a) + b; }
__device__ __forceinline__ F2 operator-(F2 a, float b) { return a - F2(b); }
__device__ __forceinline__ F2 operator-(float a, F2 b) { return F2(a) - b; }
__device__ __forceinline__ F2 operator*(F2 a, float b) { return a * F2(b); }
__device__ __forceinline__ F2 operator*(float a, F2 b) { return F2(a) * b; }

// Fused multiply-add a b + c, one rounding, for the scalar types and the pair.
__device__ __forceinline__ float vfma(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double vfma(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ F2 vfma(F2 a, F2 b, F2 c) {
  unsigned long long r;
  asm("fma.rn.ftz.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(f2_pack(a)), "l"(f2_pack(b)), "l"(f2_pack(c)));
  return f2_unpack(r);
}
__device__ __forceinline__ F2 vfma(F2 a, float b, F2 c) { return vfma(a, F2(b), c); }
__device__ __forceinline__ F2 vfma(float a, F2 b, F2 c) { return vfma(F2(a), b, c); }

// Hardware reciprocal (1 ulp; denormal arguments are flushed to zero and give an infinity).
__device__ __forceinline__ float rcp_approx(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// Componentwise operations, with the scalar overloads used by code written for either type.
__device__ __forceinline__ F2 frcp(F2 a) { return F2(rcp_approx(a.x), rcp_approx(a.y)); }
__device__ __forceinline__ float vsqrt(float a) { return sqrtf(a); }
__device__ __forceinline__ double vsqrt(double a) { return ::sqrt(a); }
__device__ __forceinline__ F2 vsqrt(F2 a) { return F2(sqrtf(a.x), sqrtf(a.y)); }
__device__ __forceinline__ float vmin(float a, float b) { return fminf(a, b); }
__device__ __forceinline__ F2 vmin(F2 a, F2 b) { return F2(fminf(a.x, b.x), fminf(a.y, b.y)); }
__device__ __forceinline__ float vmax(float a, float b) { return fmaxf(a, b); }
__device__ __forceinline__ F2 vmax(F2 a, F2 b) { return F2(fmaxf(a.x, b.x), fmaxf(a.y, b.y)); }
__device__ __forceinline__ double vmin(double a, double b) { return fmin(a, b); }
__device__ __forceinline__ double vmax(double a, double b) { return fmax(a, b); }
// The limited difference of the MC limiter from the one-sided differences dl, dr and the centred
// one q: the least of m|dl|, m|dr| and |q| with their common sign, zero where the signs of dl and dr
// differ or one is zero (q has their sign where they agree).  In FP32 three instructions per value:
// min.xorsign.abs gives the least magnitude, negative where the signs differ, which the maximum
// with zero removes; the second one gives the sign of q.  In FP64 the magnitudes and signs are
// compared as integers, which leaves the FP64 pipe to the arithmetic.
__device__ __forceinline__ float min_xs(float a, float b) {
  float y;
  asm("min.ftz.xorsign.abs.f32 %0, %1, %2;" : "=f"(y) : "f"(a), "f"(b));
  return y;
}
__device__ __forceinline__ F2 mc_min(F2 dl, F2 dr, F2 q, float m) {
  F2 r(fmaxf(min_xs(dl.x, dr.x), 0.0f), fmaxf(min_xs(dl.y, dr.y), 0.0f));
  if (m != 1.0f) r = r * m;
  return F2(min_xs(r.x, q.x), min_xs(r.y, q.y));
}
__device__ __forceinline__ double mc_min(double dl, double dr, double q, double m) {
  const long long a = __double_as_longlong(dl), b = __double_as_longlong(dr), M = 0x7fffffffffffffffLL;
  long long r = min(a & M, b & M);
  if (m != 1.0) r = __double_as_longlong(__longlong_as_double(r) * m);
  r = min(r, __double_as_longlong(q) & M);
  return (a ^ b) < 0 ? 0.0 : __longlong_as_double(r | (a & ~M));
}

// A value of type V from the values of the lane's two groups (the pair, or the first value), and
// component j of a value.
__device__ __forceinline__ float vpair(float a, float, float) { return a; }
__device__ __forceinline__ double vpair(double a, double, double) { return a; }
__device__ __forceinline__ F2 vpair(float a, float b, F2) { return F2(a, b); }
__device__ __forceinline__ float vget(float x, int) { return x; }
__device__ __forceinline__ double vget(double x, int) { return x; }
__device__ __forceinline__ float vget(F2 x, int j) { return j ? x.y : x.x; }

// Global load of a lane's groups: one 8-byte load where the pair is aligned (vec), else one by one
// (an absent second group is zero).
__device__ __forceinline__ double ld_global_lane(const double* p, bool, bool, double) { return *p; }
__device__ __forceinline__ F2 ld_global_lane(const float* p, bool vec, bool h1, F2) {
  if (vec) {
    const float2 v = *reinterpret_cast<const float2*>(p);
    return F2(v.x, v.y);
  }
  return F2(p[0], h1 ? p[1] : 0.0f);
}
// Global store of a lane's groups: one 8-byte store where the pair is aligned (vec: both exist).
__device__ __forceinline__ void st_global_lane(double* p, double v, bool, bool) { *p = v; }
__device__ __forceinline__ void st_global_lane(float* p, F2 v, bool vec, bool h1) {
  if (vec) {
    *reinterpret_cast<float2*>(p) = make_float2(v.x, v.y);
  } else {
    p[0] = v.x;
    if (h1) p[1] = v.y;
  }
}

}  // namespace fx
