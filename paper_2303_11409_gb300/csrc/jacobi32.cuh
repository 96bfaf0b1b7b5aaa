// FP32 one-sided Jacobi rotations of complex columns in shared memory, for the fronts of the refined SVDs.
//
// A column holds its rows in pairs, (re, re, im, im): 16 bytes that one lane loads at once and that FFMA2 (two
// FP32 multiply-adds an instruction on sm_103a) takes as they are, so a rotation issues 6 arithmetic
// instructions a row pair of x or y where the (re, im) layout takes 12.  The dot products run over the first R2 pairs,
// the rotation over all Rr2 (the rows below accumulate the rotations); an odd row count is filled with zeros.
//
// Measured at 192 rows, columns in shared memory, 12 warps an SM: 44-50 cycles a rotation and SM with 8-16 lanes a
// column, 64 with 32 (the scalar part is the same for any width); FP32 arithmetic alone takes 21.  Two
// columns held against two that pass halve the bytes but not the time (52 cycles): latency binds, not bytes.
#pragma once
#include <cstdint>

namespace mps {

__device__ __forceinline__ float2 row32(const float2* col, int i) {
  const float* f = reinterpret_cast<const float*>(col) + (i >> 1) * 4 + (i & 1);
  return make_float2(f[0], f[2]);
}
__device__ __forceinline__ void set_row32(float2* col, int i, float2 v) {
  float* f = reinterpret_cast<float*>(col) + (i >> 1) * 4 + (i & 1);
  f[0] = v.x;
  f[2] = v.y;
}
__host__ __device__ inline int even32(int i) { return (i + 1) & ~1; }

using f32x2 = unsigned long long;
struct __align__(16) Rows32 { f32x2 re, im; };      // one row pair
__device__ __forceinline__ f32x2 pack2(float a, float b) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ float sum2(f32x2 v) {
  float a, b;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
  return a + b;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}

__device__ __forceinline__ float rsqrt_fast(float x) {
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;\n" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ float rcp_fast(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;\n" : "=f"(r) : "f"(x));
  return r;
}

// The Jacobi rotation of two FP32 columns with squared norms al, be and inner product (gr, gi), from their
// cosine c = |g| / (|x| |y|) and d = (be - al) / (2 |x| |y|), so that nothing is squared below the range of FP32:
// q = 1 / sqrt(c^2 + d^2), cos^2 = (1 + |d| q) / 2, sin = c q / (2 cos).  cs = cos, (u, v) = the sine times the
// phase, tg = the change of the norms, c2 = c^2.  No rotation (and c2 = 0) when c <= tol or act is false.  No branches,
// and two dependent roots past the inner product, so that the latencies of two rotations overlap.
struct Rot32 { float cs, u, v, tg, c2; };
__device__ __forceinline__ Rot32 rotation32(float al, float be, float gr, float gi, float tol2, bool act) {
  const float ra = rsqrt_fast(al), rb = rsqrt_fast(be), rab = ra * rb;
  const float d = fminf(fmaxf(0.5f * (be * rb * ra - al * ra * rb), -1e18f), 1e18f);
  const float sr = gr * rab, si = gi * rab;
  const float c2 = fmaf(sr, sr, si * si);
  act = act && c2 > tol2;
  const float q = rsqrt_fast(fmaf(d, d, c2));
  const float w = fmaf(0.5f * fabsf(d), q, 0.5f), r = rsqrt_fast(w);
  const float f = copysignf(0.5f * q * r, d);
  Rot32 R;
  R.c2 = act ? c2 : 0.f;
  R.cs = act ? w * r : 1.f;
  R.u = act ? f * sr : 0.f;
  R.v = act ? f * si : 0.f;
  R.tg = act ? f * r * c2 * (al * ra) * (be * rb) : 0.f;
  return R;
}
struct Turn32 {
  f32x2 cs, u, nu, v, nv;
  __device__ __forceinline__ explicit Turn32(const Rot32& R)
      : cs(pack2(R.cs, R.cs)), u(pack2(R.u, R.u)), nu(pack2(-R.u, -R.u)), v(pack2(R.v, R.v)), nv(pack2(-R.v, -R.v)) {}
  __device__ __forceinline__ Rows32 first(const Rows32& x, const Rows32& y) const {
    return {fma2(cs, x.re, fma2(nu, y.re, mul2(nv, y.im))), fma2(cs, x.im, fma2(nu, y.im, mul2(v, y.re)))};
  }
  __device__ __forceinline__ Rows32 second(const Rows32& x, const Rows32& y) const {
    return {fma2(cs, y.re, fma2(u, x.re, mul2(nv, x.im))), fma2(cs, y.im, fma2(u, x.im, mul2(v, x.re)))};
  }
};
struct Dot32 {
  f32x2 a = 0, b = 0, c = 0, d = 0;
  __device__ __forceinline__ void add(const Rows32& x, const Rows32& y) {
    a = fma2(x.re, y.re, a);
    b = fma2(x.im, y.im, b);
    c = fma2(x.re, y.im, c);
    d = fma2(x.im, y.re, d);
  }
  __device__ __forceinline__ float2 value(int G) const {      // over the G lanes of a group; whole warps call it
    float r = sum2(a) + sum2(b), i = sum2(c) - sum2(d);
    for (int o = G >> 1; o; o >>= 1) {
      r += __shfl_xor_sync(0xffffffffu, r, o);
      i += __shfl_xor_sync(0xffffffffu, i, o);
    }
    return make_float2(r, i);
  }
};

// One warp: *nrm = the squared norm of a column's first R2 row pairs.
__device__ __forceinline__ void norm32(const float2* col, int R2, float* nrm) {
  const Rows32* a = reinterpret_cast<const Rows32*>(col);
  const int lane = threadIdx.x & 31;
  f32x2 s = 0, u = 0;
  for (int i = lane; i < R2; i += 32) {
    s = fma2(a[i].re, a[i].re, s);
    u = fma2(a[i].im, a[i].im, u);
  }
  float v = sum2(s) + sum2(u);
#pragma unroll
  for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if (lane == 0) *nrm = v;
}

// G lanes rotate columns p and q, both in shared memory (whole warps call it, with valid or without).  Returns
// the squared cosine, 0 when nothing was rotated.
__device__ __forceinline__ float pair32(float2* F, int R2, int Rr2, int ld, float* nrm, int p, int q, bool valid, int G,
                                        float tol, float floor2) {
  const int gl = threadIdx.x & (G - 1);
  const float al = valid ? nrm[p] : 0.f, be = valid ? nrm[q] : 0.f;
  const bool act = valid && fminf(al, be) > floor2;
  Rows32* ap = reinterpret_cast<Rows32*>(F + (act ? p : 0) * ld);
  Rows32* aq = reinterpret_cast<Rows32*>(F + (act ? q : 0) * ld);
  Dot32 d;
  if (act)
#pragma unroll 4
    for (int i = gl; i < R2; i += G) d.add(ap[i], aq[i]);
  const float2 g = d.value(G);
  const Rot32 T = rotation32(al, be, g.x, g.y, tol * tol, act);
  if (T.c2 == 0.f) return 0.f;
  const Turn32 turn(T);
#pragma unroll 2
  for (int i = gl; i < Rr2; i += G) {
    const Rows32 x = ap[i], y = aq[i];
    ap[i] = turn.first(x, y);
    aq[i] = turn.second(x, y);
  }
  if (gl == 0) {
    nrm[p] = fmaxf(al - T.tg, 0.f);
    nrm[q] = be + T.tg;
  }
  return T.c2;
}

// A column that G lanes hold in registers, E row pairs a lane (Rr2 <= G E), while others pass by: a rotation
// then moves one column through shared memory instead of two.
template <int G, int E>
struct Held32 {
  Rows32 x[E];
  float al;
  __device__ __forceinline__ void load(const float2* col, int Rr2, float norm) {
    const Rows32* a = reinterpret_cast<const Rows32*>(col) + (threadIdx.x & (G - 1));
    const int left = Rr2 - (int)(threadIdx.x & (G - 1));
    al = norm;
#pragma unroll
    for (int t = 0; t < E; ++t)
      if (G * t < left) x[t] = a[G * t];
  }
  __device__ __forceinline__ void store(float2* col, int Rr2) const {
    Rows32* a = reinterpret_cast<Rows32*>(col) + (threadIdx.x & (G - 1));
    const int left = Rr2 - (int)(threadIdx.x & (G - 1));
#pragma unroll
    for (int t = 0; t < E; ++t)
      if (G * t < left) a[G * t] = x[t];
  }
  // Rotates with column col (of norm *nq) unless live is false.  Whole warps call it.  Returns the squared cosine.
  __device__ __forceinline__ float meet(float2* col, float* nq, int R2, int Rr2, bool live, float tol, float floor2) {
    const int gl = threadIdx.x & (G - 1);
    Rows32* a = reinterpret_cast<Rows32*>(col) + gl;
    const int left = Rr2 - gl, dots = R2 - gl;
    const float be = *nq;
    Rows32 y[E];
#pragma unroll
    for (int t = 0; t < E; ++t)
      if (G * t < left) y[t] = a[G * t];
    Dot32 d;
#pragma unroll
    for (int t = 0; t < E; ++t)
      if (G * t < dots) d.add(x[t], y[t]);
    const float2 g = d.value(G);
    const Rot32 T = rotation32(al, be, g.x, g.y, tol * tol, live && fminf(al, be) > floor2);
    if (T.c2 == 0.f) return 0.f;
    const Turn32 turn(T);
#pragma unroll
    for (int t = 0; t < E; ++t)
      if (G * t < left) {
        const Rows32 xo = x[t];
        x[t] = turn.first(xo, y[t]);
        a[G * t] = turn.second(xo, y[t]);
      }
    al = fmaxf(al - T.tg, 0.f);
    if (gl == 0) *nq = be + T.tg;
    return T.c2;
  }
};

}  // namespace mps
