// Refinement of the sector SVDs (K2) on the tensor cores: FP64-accurate complex products from
// exact integer slices, and a quadratically convergent correction of an FP32 SVD built on them.
//
// svd_front_kernel (k_svd.cu) leaves, per sector, the FP64 Jacobi matrix J = R^dag (n x K) and the
// rotations V of an FP32 one-sided Jacobi run on it, so that A = J V has columns orthogonal to
// about 1e-5 and V^dag V = I to about 1e-6.  What remains is to make both exact:
//     R = I - V^dag V,  S = A^dag A,
//     E_pq = (S_pq + lambda_q R_pq) / (lambda_q - lambda_p),  E_pp = (R_pp - sum_k |E_kp|^2) / 2,
//     V <- V + V E,  A <- A + A E,
// which squares the error in every step (the symmetric-eigenvalue refinement of Ogita and Aishima,
// "Iterative refinement for symmetric eigenvalue decomposition", 2018, applied to the Gram matrix
// of A without ever forming it to less than column-wise relative accuracy).  Pairs whose values are
// close are turned by the Jacobi angle instead of the quotient.  Two or three steps reach rounding;
// a sector that does not settle is left to the FP64 Jacobi sweeps.
//
// The products.  GB300's FP64 pipe does 2 FMA/clk/SM and the rest of an FP64 sweep is bound by it;
// mma.sync on BF16 does 1024 MAC/clk/SM (measured, 300 TMAC/s).  A double scaled to |x| < 2^e is the
// integer x 2^(54-e), written as 7 balanced base-256 digits; a digit is exact in BF16, a product of
// two digits is an integer of at most 14 bits, and FP32 sums of up to 7 x 128 such products stay
// below 2^24, so the tensor core adds them exactly.  Digit pairs (i, j) with i + j <= 6 are kept
// (28 products), which leaves an error of about 2^-55 of the product of the two scales, below that
// of an FP64 dot product; every 64 complex k the FP32 sums move to 64-bit integers.  The digits
// are cut while a tile is staged in shared memory, so the operands stay FP64 in global memory.
#include <algorithm>
#include <atomic>

#include "mps_internal.h"
#include "refine_fixed.cuh"
#include "refine_pair.cuh"

namespace mps {
namespace {

constexpr int kOzSlices = 7;
constexpr int kOzM = 64, kOzN = 32, kOzK = 32;      // complex rows, columns and contraction of a stage
constexpr int kOzThreads = 256;                     // 4 x 2 warps of 16 x 16 complex outputs
constexpr int kOzABytes = kOzM * 128, kOzBBytes = kOzN * 128;   // one slice: 32 complex BF16 pairs a row
constexpr int kOzAhead = 4;                         // operand loads in flight ahead of their conversion
constexpr int kOzSmem = kOzSlices * (kOzABytes + kOzBBytes);

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// The slices of one complex number into its row: word = (BF16 re, BF16 im), neg flips im.
template <int NS, typename T2>
__device__ __forceinline__ void oz_store(char* base, int slice_bytes, T2 v, int e, uint32_t neg) {
  const uint64_t a = oz_fixed(v.x, e), b = oz_fixed(v.y, e);
  const uint32_t al = (uint32_t)a, ah = (uint32_t)(a >> 32), bl = (uint32_t)b, bh = (uint32_t)(b >> 32);
#pragma unroll
  for (int i = 0; i < NS; ++i) {
    const int byte = 6 - i;
    const uint32_t sel = 0x7540u | (byte & 3);
    const float fr = __uint_as_float(__byte_perm(byte >= 4 ? ah : al, 0x4B000000u, sel)) - 8388736.0f;
    const float fi = __uint_as_float(__byte_perm(byte >= 4 ? bh : bl, 0x4B000000u, sel)) - 8388736.0f;
    *reinterpret_cast<uint32_t*>(base + i * slice_bytes) =
        __byte_perm(__float_as_uint(fr), __float_as_uint(fi), 0x7632) ^ neg;
  }
}

__device__ __forceinline__ void ldsm4(uint32_t* r, uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr));
}
__device__ __forceinline__ void mma_bf16(float* c, const uint32_t* a, uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
      "{%0, %1, %2, %3};\n"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// (re, im) -> (im, -re): the operand column of the imaginary part
__device__ __forceinline__ uint32_t turn(uint32_t v) { return ((v >> 16) | (v << 16)) ^ 0x80000000u; }

// Exact sums of a warp's 16 x 16 complex tile: value = (hi 2^32 + lo) 2^(ea + eb - 60).
// Index [h][x]: column group h (8 columns), x = 0..1 row g, 2..3 row g + 8, columns 2t, 2t + 1.
struct OzSum {
  long long hi[2][2][4], lo[2][2][4];      // [re / im][h][x]
};

// One stage in shared memory: the MMAs of its k-steps (8 complex each, at most 4) into acc[slice sum][re/im * 2 + h][4].
template <int NS>
__device__ __forceinline__ void oz_stage(float (&acc)[NS][4][4], uint32_t sA, uint32_t sB, int wr, int wc, int lane,
                                         int steps) {
  const int arow = wr * 16 + (lane & 15), brow = wc * 16 + (lane & 7) + ((lane >> 4) << 3);
#pragma unroll 1
  for (int s = 0; s < steps; ++s) {
    uint32_t a[NS][4];
    const int ac = (2 * s + (lane >> 4)) ^ (arow & 7), bc = (2 * s + ((lane >> 3) & 1)) ^ (brow & 7);
#pragma unroll
    for (int i = 0; i < NS; ++i) ldsm4(a[i], sA + i * kOzABytes + arow * 128 + ac * 16);
#pragma unroll
    for (int j = 0; j < NS; ++j) {
      uint32_t b[4];
      ldsm4(b, sB + j * kOzBBytes + brow * 128 + bc * 16);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const uint32_t i0 = turn(b[2 * h]), i1 = turn(b[2 * h + 1]);
#pragma unroll
        for (int i = 0; i + j < NS; ++i) {
          mma_bf16(acc[i + j][h], a[i], b[2 * h], b[2 * h + 1]);
          mma_bf16(acc[i + j][2 + h], a[i], i0, i1);
        }
      }
    }
  }
}

template <int NS>
__device__ __forceinline__ void oz_flush(float (&acc)[NS][4][4], OzSum& t) {
#pragma unroll
  for (int z = 0; z < 4; ++z)
#pragma unroll
    for (int x = 0; x < 4; ++x) {
      long long hi = 0, lo = 0;
#pragma unroll
      for (int d = 0; d < NS; ++d) {
        const long long v = __float2int_rn(acc[d][z][x]);
        if (d < 3) hi += v << (16 - 8 * d);
        else lo += v << (48 - 8 * d);
        acc[d][z][x] = 0.f;
      }
      t.hi[z >> 1][z & 1][x] += hi;
      t.lo[z >> 1][z & 1][x] += lo;
    }
}

// t = sum over k < kt of (the A tile)(row, k)^* (the B tile)(col, k); load_a(k0) and load_b(k0) put the
// slices of stage [k0, k0 + 32) into shared memory (zero beyond kt up to a k-step).  A warp whose
// outputs are not wanted (on == false) only helps to load.
template <int NS, class LA, class LB>
__device__ void oz_product(OzSum& t, char* smem, int kt, bool on, LA load_a, LB load_b) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, wr = warp & 3, wc = warp >> 2;
  const uint32_t sA = smem_u32(smem), sB = sA + kOzSlices * kOzABytes;
  float acc[NS][4][4];
#pragma unroll
  for (int d = 0; d < NS; ++d)
#pragma unroll
    for (int z = 0; z < 4; ++z)
#pragma unroll
      for (int x = 0; x < 4; ++x) acc[d][z][x] = 0.f;
#pragma unroll
  for (int z = 0; z < 2; ++z)
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
      for (int x = 0; x < 4; ++x) t.hi[z][h][x] = t.lo[z][h][x] = 0;
  int held = 0;
  for (int k0 = 0; k0 < kt; k0 += kOzK) {
    __syncthreads();
    load_a(k0);
    load_b(k0);
    __syncthreads();
    if (!on) continue;
    oz_stage<NS>(acc, sA, sB, wr, wc, lane, (min(kOzK, kt - k0) + 7) / 8);
    if (++held == 2) {      // 64 complex k: the FP32 sums are still exact
      oz_flush<NS>(acc, t);
      held = 0;
    }
  }
  if (held) oz_flush<NS>(acc, t);
}

__device__ __forceinline__ double pow2(int e) { return __longlong_as_double((long long)(max(e, -1020) + 1023) << 52); }
__device__ __forceinline__ double oz_double(long long hi, long long lo, int e) {
  return fma((double)hi, 4294967296.0, (double)lo) * pow2(e);
}
// the same as an FP32 number in units of 2^60 (the scales taken out)
__device__ __forceinline__ float oz_float(long long hi, long long lo) {
  const float u = 8.673617379884035e-19f;      // 2^-60
  hi += lo >> 32;                               // the whole sum as (hi, 32 low bits)
  lo &= 0xffffffffLL;
  if (hi > -(1LL << 30) && hi < (1LL << 30)) return (float)((hi << 32) + lo) * u;
  return (float)hi * (4294967296.0f * u);
}

// Loaders.  A Gram operand: column c0 + row of X (column-major, ld), contraction along the column.
template <int NS, int ROWS, typename T2>
__device__ __forceinline__ void load_cols(char* dst, int slice_bytes, const T2* X, int64_t ld, int c0, int ncol, int k0,
                                          int kn, const int* e_sh) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (lane >= (min(kOzK, kn - k0) + 7) / 8 * 8) return;
  const int rows = min(ROWS, ncol - c0);
#pragma unroll 1
  for (int r0 = warp; r0 < rows; r0 += kOzAhead * kOzThreads / 32) {
    T2 v[kOzAhead];
#pragma unroll
    for (int a = 0; a < kOzAhead; ++a) {
      const int r = r0 + a * kOzThreads / 32;
      v[a].x = 0;
      v[a].y = 0;
      if (r < rows && k0 + lane < kn) v[a] = X[(int64_t)(c0 + r) * ld + k0 + lane];
    }
#pragma unroll
    for (int a = 0; a < kOzAhead; ++a) {
      const int r = r0 + a * kOzThreads / 32;
      if (r < rows)
        oz_store<NS>(dst + r * 128 + (((lane >> 2) ^ (r & 7)) << 4) + ((lane & 3) << 2), slice_bytes, v[a], e_sh[r], 0u);
    }
  }
}
// The left operand of X W: rows r0.. of X (column-major), contraction over its columns k with the
// scale exponents e[k]; conjugated, since the product conjugates its left operand.
template <int NS>
__device__ __forceinline__ void load_rows(char* dst, const double2* X, int64_t ld, int r0, int nrow, int k0, int kn,
                                          const int* e) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nr = (min(kOzM, nrow - r0) + 7) / 8, nb = (min(kOzK, kn - k0) + 7) / 8 * 2;      // 8 rows x 4 k each
#pragma unroll 1
  for (int t0 = warp; t0 < nr * nb; t0 += kOzAhead * kOzThreads / 32) {
    double2 v[kOzAhead];
    int ek[kOzAhead];
#pragma unroll
    for (int a = 0; a < kOzAhead; ++a) {
      const int t = t0 + a * kOzThreads / 32;
      const int r = (t % nr) * 8 + (lane & 7), k = 4 * (t / nr) + (lane >> 3);
      v[a] = make_double2(0.0, 0.0);
      ek[a] = 0;
      if (t < nr * nb && k0 + k < kn) {
        ek[a] = e[k0 + k];
        if (r0 + r < nrow) v[a] = X[(int64_t)(k0 + k) * ld + r0 + r];
      }
    }
#pragma unroll
    for (int a = 0; a < kOzAhead; ++a) {
      const int t = t0 + a * kOzThreads / 32, r = (t % nr) * 8 + (lane & 7), b = t / nr;
      if (t < nr * nb)
        oz_store<NS>(dst + r * 128 + ((b ^ (r & 7)) << 4) + ((lane >> 3) << 2), kOzABytes, v[a], ek[a], 0x80000000u);
    }
  }
}

// Two or three steps settle a sector; launches beyond that find nothing to do (3 us each), and what is
// not settled after the last one costs FP64 sweeps, which large sectors can least afford.
__host__ __device__ constexpr int refine_steps(int K) { return K < 200 ? 4 : kRefineSteps; }
__device__ __forceinline__ int ns_of(const SvdSector& S) { return __ldg(S.rstate); }
__device__ __forceinline__ bool skip(const SvdSector& S) { return S.rstate[1] != 0 || S.rstate[2] != 0; }

// Squared norm (FP64) and scale exponent of every column of the current A (which == 0: of J), and the scale
// exponent of V's, one warp a column; and whether step `it` has settled the sector or does not contract.  The words it writes for
// that hold `it`, so that CTAs of the same launch that see them go on with their norms.
__global__ void __launch_bounds__(256) refine_norm_kernel(const SvdSector* __restrict__ secs, int which, int it) {
  const SvdSector S = secs[blockIdx.y];
  const int left = S.rstate[1], done = S.rstate[2];
  if ((left != 0 && left != kLeftAt + it) || (done != 0 && done != it)) return;
  const int K = min(S.m, S.n), n = S.n, lane = threadIdx.x & 31;
  const int ncol = which == 0 ? K : ns_of(S);
  if (it > 0 && blockIdx.x == 0 && threadIdx.x == 0) {
    const float th = __int_as_float(S.rstate[4 + it - 1]);
    if (refine_fails(th, it - 1)) S.rstate[1] = kLeftAt + it;
    else if (refine_settles(th, ncol, n)) S.rstate[2] = it;
    else if (it >= refine_steps(K)) S.rstate[1] = kLeftAt + it;      // whatever its batch has launched
  }
  const double2* X = which == 0 ? S.J : ((it & 1) ? S.A1 : S.A0);
  for (int c = blockIdx.x * 8 + (threadIdx.x >> 5); c < ncol; c += gridDim.x * 8) {
    const double2* a = X + (int64_t)c * n;
    double s0 = 0.0, s1 = 0.0;
    unsigned top = 0;             // largest biased exponent of the column
    for (int i = lane; i < n; i += 32) {
      const double2 x = a[i];
      s0 = fma(x.x, x.x, s0);
      s1 = fma(x.y, x.y, s1);
      top = max(top, max((unsigned)(__double_as_longlong(x.x) >> 52) & 0x7ffu,
                         (unsigned)(__double_as_longlong(x.y) >> 52) & 0x7ffu));
    }
    s0 += s1;
    unsigned vtop = 0;
    if (which == 1) {
      const double2* v = ((it & 1) ? S.V1 : S.V0) + (int64_t)c * K;
      for (int k = lane; k < K; k += 32)
        vtop = max(vtop, max((unsigned)(__double_as_longlong(v[k].x) >> 52) & 0x7ffu,
                             (unsigned)(__double_as_longlong(v[k].y) >> 52) & 0x7ffu));
    }
    for (int o = 16; o; o >>= 1) {
      s0 += __shfl_xor_sync(0xffffffffu, s0, o);
      top = max(top, __shfl_xor_sync(0xffffffffu, top, o));
      vtop = max(vtop, __shfl_xor_sync(0xffffffffu, vtop, o));
    }
    if (lane == 0) {
      S.vexp[c] = max((int)vtop - 1022, -200);
      S.rnorm[c] = s0;
      S.cexp[c] = max((int)top - 1022, -900);
      if (!(s0 < 1e300)) S.rstate[1] = kLeftAt + it;      // infinities and NaN go to the FP64 sweeps
    }
  }
}

// A <- J V (step 0) or X + X E of the current [A; V] into the other buffers.
__global__ void __launch_bounds__(kOzThreads, 1) refine_update_kernel(const SvdSector* __restrict__ secs, int step) {
  extern __shared__ __align__(128) char smem[];
  __shared__ int s_t[kOzN];
  __shared__ float s_d[kOzN];      // second-order part of W's diagonal
  const SvdSector S = secs[blockIdx.y];
  if (skip(S)) return;
  const float2* E = S.E();
  const int K = min(S.m, S.n), n = S.n, ns = ns_of(S);
  const int ct = (ns + kOzN - 1) / kOzN, rtA = (n + kOzM - 1) / kOzM, rtV = step == 0 ? 0 : (K + kOzM - 1) / kOzM;
  const int tile = blockIdx.x;
  if (tile >= ct * (rtA + rtV)) return;
  const int c0 = (tile % ct) * kOzN, rt = tile / ct;
  const bool onV = rt >= rtA;
  const int r0 = (onV ? rt - rtA : rt) * kOzM, nrow = onV ? K : n;
  const int kn = step == 0 ? K : ns;
  const double2* X = step == 0 ? S.J : (onV ? ((step & 1) ? S.V0 : S.V1) : ((step & 1) ? S.A0 : S.A1));
  double2* out = step == 0 ? S.A0 : (onV ? ((step & 1) ? S.V1 : S.V0) : ((step & 1) ? S.A1 : S.A0));
  const int64_t ld = onV ? K : n;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  // scale of each column of W: the largest component of s_k W_kc, s_k the scale of X's column k.  The
  // correction E is stored in the scaled form of A's columns, s_k E_kc / s_c.
  for (int c = warp; c < kOzN; c += 8) {
    CorrectionScale cs;
    if (c0 + c < ns) {
      const int ec = step == 0 ? 0 : S.cexp[c0 + c];
      for (int k = lane; k < kn; k += 32) {
        if (step == 0) {
          const double2 w = S.V0[(int64_t)(c0 + c) * K + k];
          const int e = max((int)((__double_as_longlong(w.x) >> 52) & 0x7ff), (int)((__double_as_longlong(w.y) >> 52) & 0x7ff));
          if (e) cs.top = max(cs.top, e - 1022 + S.cexp[k]);
        } else {
          const float2 w = E[(int64_t)(c0 + c) * K + k];
          const int d = ec - S.cexp[k];      // E_kc = w 2^d
          cs.add(w.x, w.y, d, onV ? d + S.vexp[k] : 0, k == c0 + c);
        }
      }
    }
    for (int o = 16; o; o >>= 1) {
      cs.top = max(cs.top, __shfl_xor_sync(0xffffffffu, cs.top, o));
      cs.sq += __shfl_xor_sync(0xffffffffu, cs.sq, o);
      cs.diag += __shfl_xor_sync(0xffffffffu, cs.diag, o);      // one lane holds it
    }
    if (lane == 0) {
      s_d[c] = cs.second_order();
      s_t[c] = cs.scale(onV && c0 + c < ns ? S.vexp[c0 + c] : 0);
    }
  }
  __syncthreads();
  char* sB = smem + kOzSlices * kOzABytes;
  OzSum t;
  auto la = [&](int k0) { load_rows<kOzSlices>(smem, X, ld, r0, nrow, k0, kn, onV ? S.vexp : S.cexp); };
  auto lb = [&](int k0) {      // W: column c, contraction k; scaled by s_k / t_c
    if (lane >= (min(kOzK, kn - k0) + 7) / 8 * 8) return;
    const int k = k0 + lane, rows = min(kOzN, ns - c0);
    double2 vd[kOzN / 8];
    float2 vf[kOzN / 8];
#pragma unroll
    for (int a = 0; a < kOzN / 8; ++a) {
      const int r = warp + 8 * a;
      const bool in = r < rows && k < kn;
      if (step == 0) {
        vd[a] = in ? S.V0[(int64_t)(c0 + r) * K + k] : make_double2(0.0, 0.0);
      } else {
        vf[a] = in ? E[(int64_t)(c0 + r) * K + k] : make_float2(0.f, 0.f);
        if (in && k == c0 + r) vf[a].x += s_d[r];
      }
    }
    const int ek = k < kn ? S.cexp[k] : 0, ev = onV && k < kn ? S.vexp[k] : 0;
#pragma unroll
    for (int a = 0; a < kOzN / 8; ++a) {
      const int r = warp + 8 * a;
      if (r >= rows) continue;
      char* d = sB + r * 128 + (((lane >> 2) ^ (r & 7)) << 4) + ((lane & 3) << 2);
      if (step == 0) oz_store<kOzSlices>(d, kOzBBytes, vd[a], s_t[r] - ek, 0u);
      else oz_store<kOzSlices>(d, kOzBBytes, vf[a], onV ? s_t[r] - (S.cexp[c0 + r] - ek + ev) : s_t[r], 0u);
    }
  };
  const int g = lane >> 2, q = lane & 3, wr = warp & 3, wc = warp >> 2;
  const bool on = r0 + wr * 16 < nrow && c0 + wc * 16 < ns;
  oz_product<kOzSlices>(t, smem, kn, on, la, lb);
  if (!on) return;
#pragma unroll
  for (int h = 0; h < 2; ++h)
#pragma unroll
    for (int x = 0; x < 4; ++x) {
      const int i = r0 + wr * 16 + g + ((x >> 1) << 3), lc = wc * 16 + h * 8 + 2 * q + (x & 1), c = c0 + lc;
      if (i >= nrow || c >= ns) continue;
      const int e = s_t[lc] - 60 + (step == 0 || onV ? 0 : S.cexp[c]);
      double2 v = make_double2(oz_double(t.hi[0][h][x], t.lo[0][h][x], e), oz_double(t.hi[1][h][x], t.lo[1][h][x], e));
      if (step > 0) {
        const double2 o = X[(int64_t)c * ld + i];
        v.x += o.x;
        v.y += o.y;
      }
      out[(int64_t)c * ld + i] = v;
    }
}

// The correction E (scaled form) of the current A, V from S = A^dag A and R = I - V^dag V, tile by
// tile over p <= q.  rstate[4 + it] keeps the largest entry relative to its column.
__global__ void __launch_bounds__(kOzThreads, 1) refine_gram_kernel(const SvdSector* __restrict__ secs, int it) {
  extern __shared__ __align__(128) char smem[];
  __shared__ int s_ep[kOzM], s_eq[kOzN], s_vp[kOzM], s_vq[kOzN];
  const SvdSector S = secs[blockIdx.y];
  if (skip(S)) return;
  float2* E = S.E();
  const int K = min(S.m, S.n), n = S.n, ns = ns_of(S);
  const int ct = (ns + kOzN - 1) / kOzN, rt = (ns + kOzM - 1) / kOzM;
  if ((int)blockIdx.x >= ct * rt) return;
  const int p0 = (blockIdx.x / ct) * kOzM, q0 = (blockIdx.x % ct) * kOzN;
  if (p0 >= q0 + kOzN) return;                 // below the diagonal
  const double2* A = (it & 1) ? S.A1 : S.A0;
  const double2* V = (it & 1) ? S.V1 : S.V0;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (tid < kOzM) {
    s_ep[tid] = p0 + tid < ns ? S.cexp[p0 + tid] : 0;
    s_vp[tid] = p0 + tid < ns ? S.vexp[p0 + tid] : 0;
  }
  if (tid < kOzN) {
    s_eq[tid] = q0 + tid < ns ? S.cexp[q0 + tid] : 0;
    s_vq[tid] = q0 + tid < ns ? S.vexp[q0 + tid] : 0;
  }
  __syncthreads();
  char* sB = smem + kOzSlices * kOzABytes;
  const int g = lane >> 2, qq = lane & 3, wr = warp & 3, wc = warp >> 2;
  const bool on = p0 + wr * 16 < ns && q0 + wc * 16 < ns && p0 + wr * 16 < q0 + wc * 16 + 16;
  OzSum t;
  oz_product<kOzSlices>(
      t, smem, K, on, [&](int k0) { load_cols<kOzSlices, kOzM>(smem, kOzABytes, V, K, p0, ns, k0, K, s_vp); },
      [&](int k0) { load_cols<kOzSlices, kOzN>(sB, kOzBBytes, V, K, q0, ns, k0, K, s_vq); });
  float Rr[2][4], Ri[2][4];
#pragma unroll
  for (int h = 0; h < 2; ++h)
#pragma unroll
    for (int x = 0; x < 4; ++x) {
      const int p = p0 + wr * 16 + g + ((x >> 1) << 3), q = q0 + wc * 16 + h * 8 + 2 * qq + (x & 1);
      // 1 - |v_p|^2 on the diagonal is taken in integers: 1 is 2^(60 - 2 e) in the units of the sum
      const int ep = s_vp[wr * 16 + g + ((x >> 1) << 3)], eq = s_vq[wc * 16 + h * 8 + 2 * qq + (x & 1)];
      const float f = -exp2f((float)(ep + eq));
      Rr[h][x] = f * oz_float(t.hi[0][h][x] - (p == q ? 1LL << (28 - 2 * max(ep, -16)) : 0), t.lo[0][h][x]);
      Ri[h][x] = f * oz_float(t.hi[1][h][x], t.lo[1][h][x]);
    }
  oz_product<kOzSlices>(
      t, smem, n, on, [&](int k0) { load_cols<kOzSlices, kOzM>(smem, kOzABytes, A, n, p0, ns, k0, n, s_ep); },
      [&](int k0) { load_cols<kOzSlices, kOzN>(sB, kOzBBytes, A, n, q0, ns, k0, n, s_eq); });
  if (!on) return;
  float worst = 0.f;
  const double floor2 = S.rfloor2[0];
  const float tol = 2.2204460e-16f * (float)max(n, 32);
#pragma unroll
  for (int h = 0; h < 2; ++h)
#pragma unroll
    for (int x = 0; x < 4; ++x) {
      const int p = p0 + wr * 16 + g + ((x >> 1) << 3), q = q0 + wc * 16 + h * 8 + 2 * qq + (x & 1);
      if (p >= ns || q >= ns || p > q) continue;
      if (p == q) {
        E[(int64_t)q * K + p] = make_float2(0.5f * Rr[h][x], 0.f);
        worst = fmaxf(worst, fabsf(Rr[h][x]));
        continue;
      }
      const double np = S.rnorm[p], nq = S.rnorm[q];
      float2 epq = make_float2(0.f, 0.f), eqp = epq;      // scaled: s_p E_pq / s_q, s_q E_qp / s_p
      if (fmin(np, nq) > floor2) {                        // columns at the floor are left alone
        const int ep = S.cexp[p], eq = S.cexp[q];
        const float al = (float)(np * pow2(-2 * ep)), be = (float)(nq * pow2(-2 * eq));
        const float rho = exp2f((float)max(-60, min(60, eq - ep)));       // s_q / s_p
        const float gr = oz_float(t.hi[0][h][x], t.lo[0][h][x]), gi = oz_float(t.hi[1][h][x], t.lo[1][h][x]);
        const RefinePair P = refine_pair(al, be, rho, gr, gi, Rr[h][x], Ri[h][x], tol);
        epq = P.pq;
        eqp = P.qp;
        worst = fmaxf(worst, P.size);
      }
      E[(int64_t)q * K + p] = epq;
      E[(int64_t)p * K + q] = eqp;
    }
  for (int o = 16; o; o >>= 1) worst = fmaxf(worst, __shfl_xor_sync(0xffffffffu, worst, o));
  if (lane == 0 && worst > 0.f) atomicMax(S.rstate + 4 + it, __float_as_int(worst));
  // NaN fails every comparison above; it is caught by the norms
}

// Singular values, their descending order and Y of the settled sectors: warp w of a CTA takes
// column c, its rank is the number of columns ahead of it.
__global__ void __launch_bounds__(256) refine_output_kernel(const SvdSector* __restrict__ secs) {
  const SvdSector S = secs[blockIdx.y];
  const int it = S.rstate[2];
  if (S.rstate[1] != 0 || it == 0) return;
  const int K = min(S.m, S.n), n = S.n, ns = ns_of(S), lane = threadIdx.x & 31;
  const double2* A = (it & 1) ? S.A1 : S.A0;
  const double floor2 = S.rfloor2[0], up = S.rfloor2[1];
  for (int c = blockIdx.x * 8 + (threadIdx.x >> 5); c < K; c += gridDim.x * 8) {
    const double v2 = c < ns ? S.rnorm[c] : 0.0;
    const double v = v2 > floor2 ? v2 : 0.0;
    int rank = 0;
    for (int j = lane; j < K; j += 32) {
      const double w2 = j < ns ? S.rnorm[j] : 0.0;
      const double w = w2 > floor2 ? w2 : 0.0;
      rank += (w > v) || (w == v && j < c);
    }
    for (int o = 16; o; o >>= 1) rank += __shfl_xor_sync(0xffffffffu, rank, o);
    const double sg = sqrt(v), inv = v > 0.0 ? 1.0 / sg : 0.0;
    if (lane == 0) S.sigma[rank] = sg * up;
    double2* y = S.Y + (int64_t)rank * n;
    const double2* a = A + (int64_t)c * n;
    for (int j = lane; j < n; j += 32) {
      double2 z = make_double2(0.0, 0.0);
      if (v > 0.0) z = make_double2(a[j].x * inv, a[j].y * inv);
      y[S.order[j]] = z;
    }
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    *S.status = it;
    if (S.path) *S.path = MPS_SVD_REFINED;
  }
}

}  // namespace

cudaError_t launch_refine(const SvdSector* d_secs, int count, int max_k, int max_n, cudaStream_t st) {
  if (count <= 0) return cudaSuccess;
  cudaError_t e;
  static std::atomic<uint64_t> done{0};
  int dev = 0;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if (dev >= 64 || !(done.load() >> dev & 1)) {
    if ((e = cudaFuncSetAttribute(refine_update_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kOzSmem)) !=
            cudaSuccess ||
        (e = cudaFuncSetAttribute(refine_gram_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kOzSmem)) !=
            cudaSuccess)
      return e;
    if (dev < 64) done.fetch_or(1ull << dev);
  }
  // the sector is blockIdx.y, which ends at 65535
  constexpr int kMaxSectors = 65535;
  for (; count > kMaxSectors; d_secs += kMaxSectors, count -= kMaxSectors)
    if ((e = launch_refine(d_secs, kMaxSectors, max_k, max_n, st)) != cudaSuccess) return e;
  auto cd = [](int a, int b) { return (a + b - 1) / b; };
  const dim3 cols(std::min(cd(max_k, 8), 64), count);
  const int ct = cd(max_k, kOzN), rk = cd(max_k, kOzM), rn = cd(max_n, kOzM);
  refine_norm_kernel<<<cols, 256, 0, st>>>(d_secs, 0, 0);
  refine_update_kernel<<<dim3(ct * rn, count), kOzThreads, kOzSmem, st>>>(d_secs, 0);
  refine_norm_kernel<<<cols, 256, 0, st>>>(d_secs, 1, 0);
  count_launch(); count_launch(); count_launch();
  const int steps = refine_steps(max_k);
  for (int it = 0; it < steps; ++it) {
    refine_gram_kernel<<<dim3(ct * rk, count), kOzThreads, kOzSmem, st>>>(d_secs, it);
    refine_update_kernel<<<dim3(ct * (rn + rk), count), kOzThreads, kOzSmem, st>>>(d_secs, it + 1);
    refine_norm_kernel<<<cols, 256, 0, st>>>(d_secs, 1, it + 1);
    count_launch(); count_launch(); count_launch();
  }
  refine_output_kernel<<<cols, 256, 0, st>>>(d_secs);
  count_launch();
  return cudaGetLastError();
}

}  // namespace mps
