// Batched per-sector SVD of the two-site update (K2), FP64, QR-preconditioned
// one-sided Jacobi.
//
// arXiv:2303.11409, Sec. II: after the U(1) split a local update needs only
// block-sparse SVDs of the submatrices Theta(c), each at most chi x chi.  Each
// sector M = diag(lambda) Theta'(c) (m x n, K = min(m, n)) is decomposed as
//   1. Householder QR with column pivoting  M P = Q R  (R: K x n, upper trapezoidal);
//   2. one-sided (Hestenes) Jacobi on the columns of R^dag (n x K):
//      R^dag U = [s_1 v_1, ..., s_K v_K], so the column norms are the singular
//      values and the normalised columns are the right singular vectors of R;
//   3. Y = P [v_1 ... v_K], the right singular vectors of M = X S Y^dag.
// Neither Q nor the rotations are accumulated: the right-canonical reassembly
// needs only S and Y.  Pivoted QR is the Drmac-Veselic preconditioner: the
// lambda-graded sectors of an MPS (singular values over 10-15 decades) need
// 20-35 plain Jacobi sweeps but 6-8 after it.
//
// Wide sectors (cluster kernels, n >= 1.25 m): R^dag has m columns of length n; an
// unpivoted Householder QR R^dag = Q2 [R2; 0] lets the sweeps rotate the columns of the
// m x m factor R2 instead (the same rotations orthogonalise both), and
// Y = P Q2 [normalised columns; 0] is formed at the end, one warp per column.
//
// Storage: M is kept row-major with an odd leading dimension ld >= n, so the QR
// rank-1 updates are coalesced (32 consecutive columns per warp) and, once R's
// rows are conjugated in place, they are the contiguous columns of R^dag.
// Sectors of FP64 updates do not run these FP64 sweeps: svd_small_kernel (one CTA) and svd_front_kernel (a
// cluster) do an unpivoted QR and FP32 sweeps, and exact products finish them, in the CTA up to kSmallK columns
// and on the tensor cores above (k_refine.cu); the kernels below take what that leaves, and the sectors
// of reduced-precision updates.  A layer of 16 updates at chi = 512 (Bose-Hubbard, L = 32) takes 72 ms with
// it, 272 ms with the FP64 sweeps; three layers at chi = 128 (L = 24) 10.2 and 61 ms, at chi = 64 (XXZ, L = 16)
// 2.6 and 6.9.
//
// GB300 runs FP64 at 2 FMA/clk/SM, so one SM per large sector would leave a
// layer waiting on its largest sectors.  Three kernels share the work:
//   jacobi_cta_kernel:           one CTA per sector, all of it in shared memory,
//                                round-robin pair ordering;
//   jacobi_cluster_block_kernel: a thread-block cluster of 2, 4, 8 (or 16) CTAs per
//                                large sector, data in L2 (ld.global.cg /
//                                st.global.cg, no stale L1 lines across SMs), block
//                                Jacobi with the block pairs of a round staged in
//                                shared memory, CTA barriers between the steps of a
//                                round and the hardware cluster barrier between rounds;
//   jacobi_cluster_kernel:       the same data placement with round-robin pairs and
//                                register-cached columns, for sectors whose blocks do
//                                not fit in shared memory.
// Column pairs of a step are shared by groups of 8, 16 or 32 lanes (an FP64 warp
// instruction costs the same at any lane count on this part, so a warp does several
// pairs at once).  A pair is rotated when |a_p^dag a_q|^2 > tol^2 |a_p|^2 |a_q|^2,
// tol = eps * max(n, 32), and both columns are above the floor: the noise level
// 32 eps |M|_F, or a higher deflation level the caller sets (SvdSector::floor_rel,
// a fraction of the truncation cutoff, and SvdSector::floor_abs, a fraction of the
// bond's previous cut); singular values at or below the floor are reported as
// exactly 0.
// Convergence is a sweep without a rotation; a sector that does not converge
// within the sweep limit reports -1.  FP64 costs a warp 64 cycles per
// instruction here, so per-pair scalar work is kept small (no square root in the
// test; at most two rsqrt, one sqrt and one division per rotation; column norms tracked through the
// exact 2x2 relations within a sweep).
#include <algorithm>
#include <cmath>
#include <type_traits>
#include <atomic>
#include <mutex>
#include <vector>

#include "mps_internal.h"
#include "jacobi32.cuh"
#include "refine_pair.cuh"

namespace mps {
namespace {

constexpr double kEps = 2.220446049250313e-16;
constexpr int kMaxCached = 16;          // rows cached in registers per lane (n <= 512)
constexpr int kMaxCluster = 16;
constexpr int kMaxTeam = 304;           // CTAs of a team: 2 on each of 152 SMs
constexpr int kSvdExpired = -2;         // a sector's status when a bounded wait ran out
constexpr int kMaxWarps = 16;
constexpr int kBlockThreads = 192;      // block-Jacobi cluster kernel: 6 warps per CTA, 2 CTAs per SM
constexpr int kMixedMinK = 192;         // default of mps_svd_mixed_min_k
constexpr int kRefineMinK = 25;         // smallest min(m, n) refined on the tensor cores
// a refined sector's FP32 sweeps end with one that found no cosine above this: it has left about the square
constexpr float kFp32Stop = 1e-3f;
constexpr int kFrontThreads = 384;      // one-CTA fronts
// largest min(m, n) refined inside one CTA: its FP64 products at 24 columns take as long (2 x 60 us) as the
// refinement's launches do beside other sectors', and grow with the cube
constexpr int kSmallK = 24;
// rows a thread loads ahead of their use in the QR's column loops (an L2 load takes some 800 cycles,
// a row's dependent FMAs 128)
constexpr int kAhead = 8;
constexpr int kStallBlocks = 1, kStallFronts = 2;      // bits of mps_svd_inject_stall
constexpr int kMaxStaged = 16;          // block pairs staged at once by one block-Jacobi CTA

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

__device__ __forceinline__ void rr_pair(int k, int r, int mp, int& p, int& q) {
  const int ring = mp - 1;
  if (k == 0) {
    p = 0;
    q = r % ring + 1;
  } else {
    p = (k + r) % ring + 1;
    q = (ring - k + r) % ring + 1;
  }
}

// Memory access policy: plain (shared memory) or L2-only (cluster, global memory).
struct PlainMem {
  static constexpr bool kCache = false;
  template <typename T> static __device__ __forceinline__ T ld(const T* p) { return *p; }
  template <typename T> static __device__ __forceinline__ void st(T* p, T v) { *p = v; }
};
struct L2Mem {
  static constexpr bool kCache = true;    // load each column pair once per round
  static __device__ __forceinline__ double2 ld(const double2* p) { return __ldcg(p); }
  static __device__ __forceinline__ double ld(const double* p) { return __ldcg(p); }
  static __device__ __forceinline__ int ld(const int* p) { return __ldcg(p); }
  static __device__ __forceinline__ void st(double2* p, double2 v) { __stcg(p, v); }
  static __device__ __forceinline__ void st(double* p, double v) { __stcg(p, v); }
  static __device__ __forceinline__ void st(int* p, int v) { __stcg(p, v); }
};

__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;\n" ::: "memory");
}
__device__ __forceinline__ unsigned cluster_rank() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;\n" : "=r"(r));
  return r;
}

struct Rot { double c, u, v; };   // c = cos, (u + i v) = sin * gamma / |gamma|

__device__ __forceinline__ void rotate_pair(double2& x, double2& y, const Rot& R) {
  // x' = c x - s conj(e) y ;  y' = s e x + c y   with s e = u + i v
  const double2 xo = x, yo = y;
  x.x = fma(R.c, xo.x, -fma(R.u, yo.x, R.v * yo.y));
  x.y = fma(R.c, xo.y, -fma(R.u, yo.y, -R.v * yo.x));
  y.x = fma(R.c, yo.x, fma(R.u, xo.x, -R.v * xo.y));
  y.y = fma(R.c, yo.y, fma(R.u, xo.y, R.v * xo.x));
}

// One warp: orthogonalise columns p, q (length R, stride ld) of the Jacobi matrix.
// nrm holds squared column norms, updated by alpha' = alpha - t|g|, beta' = beta + t|g|.
template <class Mem>
__device__ bool jacobi_pair(double2* A, int R, int ld, double* nrm, int p, int q, double tol2, double floor2) {
  const int lane = threadIdx.x & 31;
  const double alpha = Mem::ld(nrm + p), beta = Mem::ld(nrm + q);
  if (fmin(alpha, beta) <= floor2) return false;      // a noise column: nothing to orthogonalise
  double2* ap = A + (int64_t)p * ld;
  double2* aq = A + (int64_t)q * ld;
  const bool cached = Mem::kCache && R <= 32 * kMaxCached;
  double2 xs[kMaxCached], ys[kMaxCached];
  double gr = 0.0, gi = 0.0;
  if (cached) {
#pragma unroll
    for (int t = 0; t < kMaxCached; ++t) {
      const int i = lane + 32 * t;
      xs[t] = make_double2(0.0, 0.0);
      ys[t] = make_double2(0.0, 0.0);
      if (i < R) {
        xs[t] = Mem::ld(ap + i);
        ys[t] = Mem::ld(aq + i);
      }
    }
#pragma unroll
    for (int t = 0; t < kMaxCached; ++t) {
      if (32 * t < R) {
        gr = fma(xs[t].x, ys[t].x, fma(xs[t].y, ys[t].y, gr));
        gi = fma(xs[t].x, ys[t].y, fma(-xs[t].y, ys[t].x, gi));
      }
    }
  } else {
    for (int i = lane; i < R; i += 32) {
      const double2 x = Mem::ld(ap + i), y = Mem::ld(aq + i);
      gr = fma(x.x, y.x, fma(x.y, y.y, gr));
      gi = fma(x.x, y.y, fma(-x.y, y.x, gi));
    }
  }
  gr = warp_sum(gr);
  gi = warp_sum(gi);
  const double g2 = fma(gr, gr, gi * gi);
  if (!(g2 > tol2 * alpha * beta)) return false;       // orthogonal to tolerance
  // 2x2 Hermitian Gram [[alpha, gamma], [conj(gamma), beta]] -> diagonal
  const double inv_g = rsqrt(g2);
  const double g = g2 * inv_g;
  const double zeta = (beta - alpha) * (0.5 * inv_g);
  const double t = copysign(1.0, zeta) / (fabs(zeta) + sqrt(fma(zeta, zeta, 1.0)));
  Rot Rt;
  Rt.c = rsqrt(fma(t, t, 1.0));
  const double s_over_g = Rt.c * t * inv_g;
  Rt.u = s_over_g * gr;
  Rt.v = s_over_g * gi;
  if (cached) {
#pragma unroll
    for (int k = 0; k < kMaxCached; ++k) {
      const int i = lane + 32 * k;
      if (32 * k < R) {
        rotate_pair(xs[k], ys[k], Rt);
        if (i < R) {
          Mem::st(ap + i, xs[k]);
          Mem::st(aq + i, ys[k]);
        }
      }
    }
  } else {
    for (int i = lane; i < R; i += 32) {
      double2 x = Mem::ld(ap + i), y = Mem::ld(aq + i);
      rotate_pair(x, y, Rt);
      Mem::st(ap + i, x);
      Mem::st(aq + i, y);
    }
  }
  if (lane == 0) {
    const double tg = t * g;
    Mem::st(nrm + p, fmax(alpha - tg, 0.0));
    Mem::st(nrm + q, beta + tg);
  }
  return true;
}

// G lanes (G = 8, 16 or 32; groups aligned within the warp) orthogonalise columns p, q
// (length R, column c at A + c * ld) of a shared-memory matrix, so that one warp works
// on 32 / G pairs at once.  On this part every FP64 warp instruction costs the same
// whatever its lane count, so the group-wide reduction and the scalar rotation
// parameters, which all lanes of a group compute redundantly, are shared by the
// 32 / G pairs of a warp instead of being paid per pair.  Lanes of an invalid slot only
// take part in the shuffles.  The rotation follows from the 2x2 Gram matrix
// [[alpha, g], [conj g, beta]] with tau = tan(theta) / |g| = 2 sign(D) / (|D| + sqrt(D^2 + 4|g|^2)),
// D = beta - alpha, which avoids a separate 1 / |g|; norms update by -/+ tau |g|^2.
__device__ bool jacobi_pair_grp(double2* A, int R, int ld, double* nrm, int p, int q, bool valid, int G,
                                double tol2, double floor2) {
  const int gl = threadIdx.x & (G - 1);
  double alpha = 0.0, beta = 0.0;
  if (valid) {
    alpha = nrm[p];
    beta = nrm[q];
  }
  bool act = valid && fmin(alpha, beta) > floor2;   // noise columns are left alone
  double2* ap = A + (int64_t)(act ? p : 0) * ld;
  double2* aq = A + (int64_t)(act ? q : 0) * ld;
  // two independent partial sums per component halve the FP64 dependency chains (the
  // FP64 pipe's latency, not its issue rate, bounds a lone chain)
  double gr = 0.0, gi = 0.0;
  if (act) {
    double gr1 = 0.0, gi1 = 0.0;
    int i = gl;
    for (; i + G < R; i += 2 * G) {
      const double2 x = ap[i], y = aq[i], x1 = ap[i + G], y1 = aq[i + G];
      gr = fma(x.x, y.x, fma(x.y, y.y, gr));
      gi = fma(x.x, y.y, fma(-x.y, y.x, gi));
      gr1 = fma(x1.x, y1.x, fma(x1.y, y1.y, gr1));
      gi1 = fma(x1.x, y1.y, fma(-x1.y, y1.x, gi1));
    }
    if (i < R) {
      const double2 x = ap[i], y = aq[i];
      gr = fma(x.x, y.x, fma(x.y, y.y, gr));
      gi = fma(x.x, y.y, fma(-x.y, y.x, gi));
    }
    gr += gr1;
    gi += gi1;
  }
  for (int o = G >> 1; o; o >>= 1) {
    gr += __shfl_xor_sync(0xffffffffu, gr, o);
    gi += __shfl_xor_sync(0xffffffffu, gi, o);
  }
  const double g2 = fma(gr, gr, gi * gi);
  act = act && (g2 > tol2 * alpha * beta);           // orthogonal to tolerance otherwise
  if (act) {
    const double delta = beta - alpha;
    const double tau = copysign(2.0, delta) / (fabs(delta) + sqrt(fma(delta, delta, 4.0 * g2)));
    Rot Rt;
    Rt.c = rsqrt(fma(tau * tau, g2, 1.0));
    const double ct = Rt.c * tau;
    Rt.u = ct * gr;
    Rt.v = ct * gi;
#pragma unroll 2
    for (int i = gl; i < R; i += G) {
      double2 x = ap[i], y = aq[i];
      rotate_pair(x, y, Rt);
      ap[i] = x;
      aq[i] = y;
    }
    if (gl == 0) {
      const double tg = tau * g2;
      nrm[p] = fmax(alpha - tg, 0.0);
      nrm[q] = beta + tg;
    }
  }
  return act;
}

// Group width for P disjoint pairs of columns of length R spread over nwarps warps:
// the width with the fewest FP64 warp instructions per warp, counting the passes
// needed (ceil(P / slots)) times the instructions of one pass (about 16 per column
// element a lane holds, plus about 50 for the reduction and the rotation parameters).
__device__ __forceinline__ int group_width(int P, int R, int nwarps) {
  int best = 32;
  long long best_cost = -1;
  for (int G = 32; G >= 8; G >>= 1) {
    const int slots = nwarps * (32 / G);
    const long long cost = (long long)((P + slots - 1) / slots) * (16 * ((R + G - 1) / G) + 50);
    if (best_cost < 0 || cost < best_cost) { best_cost = cost; best = G; }
  }
  return best;
}

// The same for a group of G = 32 wg lanes (wg > 1 whole warps, groups aligned to wg warps)
// per pair, for steps with fewer disjoint pairs than warps (the large sectors, whose column
// blocks hold only 3-5 columns): each warp reduces its part of the dot product with shuffles
// and the group sums the warp partials through shared memory behind a named barrier (id
// bar_id, one per group).  red holds two buffers of 2 doubles per warp, used alternately
// (phase), so a warp that runs ahead into the next pair never overwrites partials still read.
__device__ bool jacobi_pair_mw(double2* A, int R, int ld, double* nrm, int p, int q, bool valid, int G,
                               double tol2, double floor2, double* red, int& phase, int bar_id) {
  const int wg = G >> 5, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int w0 = warp - warp % wg, gl = (warp - w0) * 32 + lane;
  double* rb = red + phase * 2 * kMaxWarps;
  phase ^= 1;
  double alpha = 0.0, beta = 0.0;
  if (valid) {
    alpha = nrm[p];
    beta = nrm[q];
  }
  bool act = valid && fmin(alpha, beta) > floor2;
  double2* ap = A + (int64_t)(act ? p : 0) * ld;
  double2* aq = A + (int64_t)(act ? q : 0) * ld;
  double gr = 0.0, gi = 0.0;
  if (act) {
    double gr1 = 0.0, gi1 = 0.0;
    int i = gl;
    for (; i + G < R; i += 2 * G) {
      const double2 x = ap[i], y = aq[i], x1 = ap[i + G], y1 = aq[i + G];
      gr = fma(x.x, y.x, fma(x.y, y.y, gr));
      gi = fma(x.x, y.y, fma(-x.y, y.x, gi));
      gr1 = fma(x1.x, y1.x, fma(x1.y, y1.y, gr1));
      gi1 = fma(x1.x, y1.y, fma(-x1.y, y1.x, gi1));
    }
    if (i < R) {
      const double2 x = ap[i], y = aq[i];
      gr = fma(x.x, y.x, fma(x.y, y.y, gr));
      gi = fma(x.x, y.y, fma(-x.y, y.x, gi));
    }
    gr += gr1;
    gi += gi1;
  }
  gr = warp_sum(gr);
  gi = warp_sum(gi);
  if (lane == 0) {
    rb[2 * warp] = gr;
    rb[2 * warp + 1] = gi;
  }
  asm volatile("bar.sync %0, %1;\n" ::"r"(bar_id), "r"(G) : "memory");
  gr = 0.0;
  gi = 0.0;
  for (int x = 0; x < wg; ++x) {        // the same order in every warp of the group
    gr += rb[2 * (w0 + x)];
    gi += rb[2 * (w0 + x) + 1];
  }
  const double g2 = fma(gr, gr, gi * gi);
  act = act && (g2 > tol2 * alpha * beta);
  if (act) {
    const double delta = beta - alpha;
    const double tau = copysign(2.0, delta) / (fabs(delta) + sqrt(fma(delta, delta, 4.0 * g2)));
    Rot Rt;
    Rt.c = rsqrt(fma(tau * tau, g2, 1.0));
    const double ct = Rt.c * tau;
    Rt.u = ct * gr;
    Rt.v = ct * gi;
#pragma unroll 2
    for (int i = gl; i < R; i += G) {
      double2 x = ap[i], y = aq[i];
      rotate_pair(x, y, Rt);
      ap[i] = x;
      aq[i] = y;
    }
    if (gl == 0) {
      const double tg = tau * g2;
      nrm[p] = fmax(alpha - tg, 0.0);
      nrm[q] = beta + tg;
    }
  }
  return act;
}

// Group width for P disjoint pairs of length R over nwarps warps, multi-warp groups
// included (wg warps per pair, wg dividing nwarps; about 40 more instructions per pass for
// the shared-memory reduction).  Returns G; slots() gives the pairs one pass covers.
__device__ __forceinline__ int group_width_mw(int P, int R, int nwarps) {
  int best = 32;
  long long best_cost = -1;
  for (int G = 8; G <= 32 * nwarps; G = (G < 32) ? 2 * G : G + 32) {
    if (G > 32 && nwarps % (G >> 5) != 0) continue;
    const int slots = G <= 32 ? nwarps * (32 / G) : nwarps / (G >> 5);
    const long long cost =
        (long long)((P + slots - 1) / slots) * (16 * ((R + G - 1) / G) + 50 + (G > 32 ? 40 : 0));
    if (best_cost < 0 || cost < best_cost) { best_cost = cost; best = G; }
  }
  return best;
}
__device__ __forceinline__ int group_slots(int G, int nwarps) { return G <= 32 ? nwarps * (32 / G) : nwarps / (G >> 5); }
__device__ __forceinline__ int group_slot(int G) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  return G <= 32 ? warp * (32 / G) + lane / G : warp / (G >> 5);
}

// Bulk copies (the TMA engine, no tensor map) of whole staged columns: a column of the Jacobi
// matrix is contiguous in global memory and in the staging area, 16-byte aligned, a multiple of
// 16 bytes long.  One thread issues them; the CTA waits on an mbarrier (loads) or the issuing
// thread on the bulk group (stores).  Global data crosses between the generic and the async
// proxy only behind fence.proxy.async and the cluster barrier, staged data behind the same fence for
// shared memory and a CTA barrier.
__device__ __forceinline__ uint32_t sh_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void stage_bar_init(uint64_t* b) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(sh_addr(b)) : "memory");
  asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
}
__device__ __forceinline__ void stage_expect(uint64_t* b, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(sh_addr(b)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes, uint64_t* b) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(
                   sh_addr(dst)),
               "l"(src), "r"(bytes), "r"(sh_addr(b))
               : "memory");
}
__device__ __forceinline__ void bulk_store(void* dst, const void* src, uint32_t bytes) {
  asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;\n" ::"l"(dst), "r"(sh_addr(src)),
               "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void bulk_store_drain() {
  asm volatile("cp.async.bulk.commit_group;\n" ::: "memory");
  asm volatile("cp.async.bulk.wait_group 0;\n" ::: "memory");
  asm volatile("fence.proxy.async.global;\n" ::: "memory");
}
__device__ __forceinline__ void fence_to_async() { asm volatile("fence.proxy.async.global;\n" ::: "memory"); }
// Every thread, between its accesses of staged columns and the barrier before a bulk copy reads or overwrites them.
__device__ __forceinline__ void fence_stage() { asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory"); }
// Bounded wait (about 2 s; 50 ms when the barrier is made to expect bytes that never come) for the
// staging barrier's phase; false when it expired.  The CTA then leaves its columns alone, keeps to the
// barriers that it shares with others, and waits once more for its copies in flight before it ends.
__device__ __forceinline__ bool stage_wait(uint64_t* b, uint32_t parity, bool stall) {
  const long long limit = stall ? 100000000LL : 4000000000LL;
  const uint32_t a = sh_addr(b);
  const long long t0 = clock64();
  for (;;) {
    uint32_t done;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(a), "r"(parity)
        : "memory");
    if (done) return true;
    if (clock64() - t0 > limit) return false;
  }
}

// Per-sector working set (shared memory or global scratch).
struct Work {
  double2* W;     // m x ld, row-major: M, then R (rows 0..K-1), then R^dag's columns
  double2* u;     // m: Householder vector of the current step
  double* nu;     // n: partial squared column norms for pivoting
  double* nu0;    // n: their reference values (recompute when cancellation sets in)
  int* perm;      // n: column permutation P
  double* nrm;    // K: Jacobi column norms / singular values
  int* ord;       // K: descending order of the singular values
  int* flags;     // max_sweeps + 1: rotation seen in sweep s
  double* pv;     // per-CTA pivot candidates (value)
  int* pi;        // per-CTA pivot candidates (index)
  double* scal;   // [0] = 2 / u^dag u, [1] = |M|_F^2
};

__host__ __device__ inline int odd_ld(int n) { return n | 1; }

// Round-robin Jacobi sweeps: every round's disjoint pairs spread over all warps that
// share the sector, one barrier per round.
template <class Mem>
struct JacobiRoundRobin {
  static constexpr int kPath = Mem::kCache ? MPS_SVD_ROUND_ROBIN : 0;
  template <class Sync>
  __device__ int operator()(double2* W, int n, int ld, int K, const Work& w, int rank, int nctas, Sync sync,
                            double tol2, double floor2, int max_sweeps, bool& converged) const {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    const int worker = rank * nwarps + warp, workers = nctas * nwarps;
    const int mp = K + (K & 1);
    int sweep = 0;
    converged = K < 2;
    for (; !converged && sweep < max_sweeps; ++sweep) {
      if (sweep > 0) {          // fresh squared norms at the start of every sweep
        for (int j = worker; j < K; j += workers) {
          const double2* a = W + (int64_t)j * ld;
          double acc = 0.0;
          for (int i = lane; i < n; i += 32) {
            const double2 x = Mem::ld(a + i);
            acc = fma(x.x, x.x, fma(x.y, x.y, acc));
          }
          acc = warp_sum(acc);
          if (lane == 0) Mem::st(w.nrm + j, acc);
        }
        sync();
      }
      for (int r = 0; r < mp - 1; ++r) {
        bool rot = false;
        if constexpr (!Mem::kCache) {   // shared memory: several pairs per warp
          const int G = group_width(mp / 2, n, workers), per = 32 / G, slot = worker * per + lane / G;
          for (int base = 0; base < mp / 2; base += workers * per) {
            const int kk = base + slot;
            int p = 0, q = 0;
            if (kk < mp / 2) rr_pair(kk, r, mp, p, q);
            const bool valid = kk < mp / 2 && p < K && q < K;
            rot |= jacobi_pair_grp(W, n, ld, w.nrm, min(p, q), max(p, q), valid, G, tol2, floor2);
          }
          if (rot) Mem::st(w.flags + sweep, 1);
        } else {
          for (int kk = worker; kk < mp / 2; kk += workers) {
            int p, q;
            rr_pair(kk, r, mp, p, q);
            if (p >= K || q >= K) continue;
            if (p > q) { const int t = p; p = q; q = t; }
            rot |= jacobi_pair<Mem>(W, n, ld, w.nrm, p, q, tol2, floor2);
          }
          if (rot && lane == 0) Mem::st(w.flags + sweep, 1);
        }
        sync();
      }
      converged = Mem::ld(w.flags + sweep) == 0;
    }
    return sweep;
  }
};

// Block-Jacobi sweeps for a cluster sector (data in L2).  The K columns form
// nb = 2 * nctas * g contiguous blocks; in block round r the blocks are paired by the
// round-robin ordering and CTA `rank` takes the pairs rank, rank + nctas, ... (g of
// them), staging gs of them at a time (both blocks and their norms) in shared memory.
// For the staged pairs it orthogonalises, in round 0, every pair inside each block
// (round-robin inside the block) and then every cross pair (cyclic shifts of the
// larger block against the smaller), all staged block pairs advancing together so
// that each step has about gs * K / nb disjoint pairs for the warp groups; steps are
// separated by CTA barriers, the round by one cluster barrier.  Every pair is visited
// once per sweep.
struct JacobiBlocks {
  static constexpr int kPath = 0;
  double2* sm;   // 2 * gs * bsmax columns of n complex (shared memory)
  double* smn;   // 2 * gs * bsmax norms (shared memory)
  int bsmax;
  int g;         // a round has cl0 * g block pairs; CTA `rank` takes the pairs rank, rank + nctas, ...
  int gs;        // block pairs staged at once
  int cl0;       // the cluster size that fixes the block ordering (nctas itself on a cluster)
  bool stall;    // expect bytes that no copy brings
  // how many block pairs a cluster's CTA stages together with pair p
  __device__ int staged_with(int p) const {
    const int q = p / cl0;
    return min(gs, g - q / gs * gs);
  }
  template <class Sync>
  __device__ int operator()(double2* W, int n, int ld, int K, const Work& w, int rank, int nctas, Sync sync,
                            double tol2, double floor2, int max_sweeps, bool& converged) const {
    __shared__ int s_rot;
    __shared__ double s_red[2 * 2 * kMaxWarps];   // multi-warp pair partials, two buffers
    __shared__ __align__(8) uint64_t s_bar;       // staging loads
    int mw_phase = 0;
    uint32_t stage_parity = 0;
    if (threadIdx.x == 0) stage_bar_init(&s_bar);
    __syncthreads();
    __shared__ int s_col[2 * kMaxStaged];   // first column of each staged block
    __shared__ int s_len[2 * kMaxStaged];   // its width (0: slot unused)
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarps = blockDim.x >> 5;
    const int worker = rank * nwarps + warp, workers = nctas * nwarps;
    const int nb = 2 * cl0 * g, own = (cl0 * g - rank + nctas - 1) / nctas;
    const bool team = nctas != cl0;   // one pair at a time, in the lane groups the cluster would use
    bool dead = false;                // a wait of this CTA expired
    int sweep = 0;
    converged = K < 2;
    for (; !converged && sweep < max_sweeps; ++sweep) {
      if (sweep > 0) {
        for (int j = worker; j < K; j += workers) {
          const double2* a = W + (int64_t)j * ld;
          double acc = 0.0;
          for (int i = lane; i < n; i += 32) {
            const double2 x = __ldcg(a + i);
            acc = fma(x.x, x.x, fma(x.y, x.y, acc));
          }
          acc = warp_sum(acc);
          if (lane == 0) __stcg(w.nrm + j, acc);
        }
        sync();
      }
      if (tid == 0) s_rot = 0;
      bool rot = false;
      for (int r = 0; r < nb - 1; ++r) {
        for (int c0 = 0; c0 < own && !dead; c0 += team ? 1 : gs) {        // chunks of gs block pairs of this CTA
          const int ns = team ? 1 : min(gs, g - c0);
          const int ns_ref = team ? staged_with(rank + c0 * nctas) : ns;
          if (tid < 2 * gs) {
            const int j = tid >> 1;
            int col = 0, len = 0;
            if (j < ns) {
              int bp, bq;
              rr_pair(rank + (c0 + j) * nctas, r, nb, bp, bq);
              const int b = (tid & 1) ? bq : bp;
              col = (int)((int64_t)K * b / nb);
              len = (int)((int64_t)K * (b + 1) / nb) - col;
            }
            s_col[tid] = col;
            s_len[tid] = len;
          }
          __syncthreads();
          // stage: block slot j occupies columns [j * bsmax, j * bsmax + len) of sm, one bulk
          // copy per column
          if (tid == 0) {
            uint32_t bytes = 0;
            for (int j = 0; j < 2 * ns; ++j) bytes += (uint32_t)s_len[j] * (uint32_t)n * 16u;
            fence_to_async();
            stage_expect(&s_bar, bytes + (stall ? 16u : 0u));
            for (int j = 0; j < 2 * ns; ++j)
              for (int c = 0; c < s_len[j]; ++c)
                bulk_load(sm + ((int64_t)j * bsmax + c) * n, W + (int64_t)(s_col[j] + c) * ld, (uint32_t)n * 16u,
                          &s_bar);
          }
          for (int j = 0; j < 2 * ns; ++j)
            for (int c = tid; c < s_len[j]; c += blockDim.x) smn[j * bsmax + c] = __ldcg(w.nrm + s_col[j] + c);
          dead = __syncthreads_or(!stage_wait(&s_bar, stage_parity, stall));
          if (dead) break;
          stage_parity ^= 1u;
          if (r == 0) {   // pairs inside each staged block, round-robin within the block
            const int mpb = bsmax + (bsmax & 1);
            const int P = 2 * ns * (mpb / 2);
            const int G = group_width_mw(2 * ns_ref * (mpb / 2), n, nwarps), slots = group_slots(G, nwarps), slot = group_slot(G);
            for (int rr = 0; rr < mpb - 1; ++rr) {
              for (int base = 0; base < P; base += slots) {
                const int k = base + slot, j = k / (mpb / 2);
                int a = 0, b = 0;
                bool valid = k < P;
                if (valid) {
                  rr_pair(k % (mpb / 2), rr, mpb, a, b);
                  valid = a < s_len[j] && b < s_len[j];
                }
                if (G <= 32)
                  rot |= jacobi_pair_grp(sm, n, n, smn, j * bsmax + min(a, b), j * bsmax + max(a, b), valid, G,
                                         tol2, floor2);
                else
                  rot |= jacobi_pair_mw(sm, n, n, smn, j * bsmax + min(a, b), j * bsmax + max(a, b), valid, G,
                                        tol2, floor2, s_red, mw_phase, 1 + slot);
              }
              __syncthreads();
            }
          }
          {   // cross pairs: block slots 2j and 2j + 1, the smaller block shifted against the larger
            const int P = ns * bsmax;
            const int G = group_width_mw(ns_ref * bsmax, n, nwarps), slots = group_slots(G, nwarps), slot = group_slot(G);
            for (int t = 0; t < bsmax; ++t) {
              for (int base = 0; base < P; base += slots) {
                const int k = base + slot, j = k / bsmax, i = k % bsmax;
                int p = 0, q = 0;
                bool valid = false;
                if (k < P) {
                  const int la = s_len[2 * j], lb = s_len[2 * j + 1];
                  const bool swap = la > lb;
                  const int sa = swap ? lb : la, sb = swap ? la : lb;
                  valid = i < sa && t < sb;
                  if (valid) {
                    const int pa = (2 * j + (swap ? 1 : 0)) * bsmax + i;
                    const int pb = (2 * j + (swap ? 0 : 1)) * bsmax + (i + t) % sb;
                    p = min(pa, pb);
                    q = max(pa, pb);
                  }
                }
                if (G <= 32)
                  rot |= jacobi_pair_grp(sm, n, n, smn, p, q, valid, G, tol2, floor2);
                else
                  rot |= jacobi_pair_mw(sm, n, n, smn, p, q, valid, G, tol2, floor2, s_red, mw_phase, 1 + slot);
              }
              if (t + 1 == bsmax) fence_stage();
              __syncthreads();
            }
          }
          if (tid == 0) {   // write the staged columns back, one bulk copy each
            for (int j = 0; j < 2 * ns; ++j)
              for (int c = 0; c < s_len[j]; ++c)
                bulk_store(W + (int64_t)(s_col[j] + c) * ld, sm + ((int64_t)j * bsmax + c) * n, (uint32_t)n * 16u);
            bulk_store_drain();
          }
          for (int j = 0; j < 2 * ns; ++j)
            for (int c = tid; c < s_len[j]; c += blockDim.x) __stcg(w.nrm + s_col[j] + c, smn[j * bsmax + c]);
          __syncthreads();   // the next chunk reuses the staging buffers and block tables
        }
        sync();
      }
      if (rot) s_rot = 1;
      __syncthreads();
      if (tid == 0 && s_rot) __stcg(w.flags + sweep, 1);
      if (tid == 0 && dead) __stcg(w.flags + max_sweeps, 1);
      sync();
      converged = __ldcg(w.flags + sweep) == 0;
      if (__ldcg(w.flags + max_sweeps) != 0) {      // some CTA's wait
        if (dead) stage_wait(&s_bar, stage_parity, stall);
        return kSvdExpired;
      }
    }
    return sweep;
  }
};

// ---------------------------------------------------------------------------------------
// Mixed-precision preconditioning of a cluster sector (after Gao, Ma and Shao, "A mixed
// precision Jacobi SVD algorithm", 2022).  The Jacobi matrix J (jlen x K, FP64) is rounded to
// FP32 and stacked on the identity, F = [fl32(J); I]; FP32 one-sided Jacobi sweeps rotate the
// columns of both (the dot products run over the J rows only), so that the lower block
// accumulates the rotations V.  One-sided Jacobi is column-wise relatively accurate, so J V has
// relatively orthogonal columns to about FP32 precision even for columns 10-15 decades below
// the largest.  The columns whose FP32 norm is above a tenth of the deflation floor are kept,
// V is made unitary in FP64 by one Cholesky QR (V^dag V = U^dag U, V <- V U^-1; V is unitary to
// about 1e-5, so one pass leaves it unitary to rounding), and A1 = J V (FP64) starts the FP64
// sweeps, which then converge in 2-3 sweeps instead of 7-12.  The singular values of A1 are
// those of J (V unitary), and the FP64 sweeps make them and the vectors FP64-accurate; columns
// left out lie below the floor anyway.  FP32 runs at 64x the FP64 rate on this part.
// ---------------------------------------------------------------------------------------
__device__ __forceinline__ float warp_sum_f(float v) {
#pragma unroll
  for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// G lanes (8, 16 or 32) orthogonalise columns p, q of an FP32 matrix: the dot product over the
// first R rows, the rotation over the first Rr rows.  Tests and parameters avoid squaring the
// (possibly tiny) inner product: |g| against tol sqrt(alpha beta), t = tan(theta) from
// zeta = (beta - alpha) / (2 |g|).
__device__ bool jacobi_pair32(float2* A, int R, int Rr, int ld, float* nrm, int p, int q, bool valid, int G,
                              float tol, float floor2) {
  const int gl = threadIdx.x & (G - 1);
  float alpha = 0.f, beta = 0.f;
  if (valid) {
    alpha = nrm[p];
    beta = nrm[q];
  }
  bool act = valid && fminf(alpha, beta) > floor2;
  float2* ap = A + (int64_t)(act ? p : 0) * ld;
  float2* aq = A + (int64_t)(act ? q : 0) * ld;
  float gr = 0.f, gi = 0.f;
  if (act)
    for (int i = gl; i < R; i += G) {
      const float2 x = ap[i], y = aq[i];
      gr = fmaf(x.x, y.x, fmaf(x.y, y.y, gr));
      gi = fmaf(x.x, y.y, fmaf(-x.y, y.x, gi));
    }
  for (int o = G >> 1; o; o >>= 1) {
    gr += __shfl_xor_sync(0xffffffffu, gr, o);
    gi += __shfl_xor_sync(0xffffffffu, gi, o);
  }
  const float ag = hypotf(gr, gi);
  act = act && (ag > tol * sqrtf(alpha) * sqrtf(beta));
  if (act) {
    const float zeta = (beta - alpha) / (2.f * ag), az = fabsf(zeta);
    const float t = copysignf(1.f, zeta) / (az + (az < 1e18f ? sqrtf(fmaf(zeta, zeta, 1.f)) : az));
    const float c = rsqrtf(fmaf(t, t, 1.f));
    const float ct = c * t / ag;
    const float u = ct * gr, v = ct * gi;
    for (int i = gl; i < Rr; i += G) {
      const float2 x = ap[i], y = aq[i];
      ap[i] = make_float2(fmaf(c, x.x, -fmaf(u, y.x, v * y.y)), fmaf(c, x.y, -fmaf(u, y.y, -v * y.x)));
      aq[i] = make_float2(fmaf(c, y.x, fmaf(u, x.x, -v * x.y)), fmaf(c, y.y, fmaf(u, x.y, v * x.x)));
    }
    if (gl == 0) {
      const float tg = t * ag;
      nrm[p] = fmaxf(alpha - tg, 0.f);
      nrm[q] = beta + tg;
    }
  }
  return act;
}

__device__ __forceinline__ int group_width32(int P, int R, int nwarps) {
  int best = 32;
  long long best_cost = -1;
  for (int G = 32; G >= 8; G >>= 1) {
    const int slots = nwarps * (32 / G);
    const long long cost = (long long)((P + slots - 1) / slots) * (2 * ((R + G - 1) / G) + 30);
    if (best_cost < 0 || cost < best_cost) { best_cost = cost; best = G; }
  }
  return best;
}

// FP32 block-Jacobi sweeps over the K columns of F (column c at F + c * ld): the same block
// ordering as JacobiBlocks, columns of Rr FP32 complex staged whole in shared memory (the
// FP64 kernel's staging area holds them: 8 (jlen + K) <= 16 jlen bytes per column), dot
// products over the first R rows.  Returns the sweeps used (converged: a sweep without a
// rotation) or kSvdExpired.  flags: max_sweeps + 1 ints, zero on entry (the last for a wait that expired).
struct JacobiBlocks32 {
  float2* sm;
  float* smn;
  int bsmax, g, gs, cl0;      // as in JacobiBlocks
  bool stall;
  __device__ int staged_with(int p) const {
    const int q = p / cl0;
    return min(gs, g - q / gs * gs);
  }
  template <class Sync>
  __device__ int operator()(float2* F, int R, int Rr, int ld, int K, float* nrm, int* flags, int rank, int nctas,
                            Sync sync, float tol, float floor2, int max_sweeps, bool& converged) const {
    __shared__ int s_rot32;
    __shared__ int s_col32[2 * kMaxStaged];
    __shared__ int s_len32[2 * kMaxStaged];
    __shared__ __align__(8) uint64_t s_bar32;
    uint32_t stage_parity = 0;
    if (threadIdx.x == 0) stage_bar_init(&s_bar32);
    __syncthreads();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarps = blockDim.x >> 5;
    const int worker = rank * nwarps + warp, workers = nctas * nwarps;
    const int nb = 2 * cl0 * g, own = (cl0 * g - rank + nctas - 1) / nctas;
    const bool team = nctas != cl0;
    bool dead = false;
    int sweep = 0;
    converged = K < 2;
    for (; !converged && sweep < max_sweeps; ++sweep) {
      for (int j = worker; j < K; j += workers) {   // fresh squared norms over the J rows
        const float2* a = F + (int64_t)j * ld;
        float acc = 0.f;
        for (int i = lane; i < R; i += 32) {
          const float2 x = __ldcg(a + i);
          acc = fmaf(x.x, x.x, fmaf(x.y, x.y, acc));
        }
        acc = warp_sum_f(acc);
        if (lane == 0) __stcg(nrm + j, acc);
      }
      sync();
      if (tid == 0) s_rot32 = 0;
      bool rot = false;
      for (int r = 0; r < nb - 1; ++r) {
        for (int c0 = 0; c0 < own && !dead; c0 += team ? 1 : gs) {
          const int ns = team ? 1 : min(gs, g - c0);
          const int ns_ref = team ? staged_with(rank + c0 * nctas) : ns;
          if (tid < 2 * gs) {
            const int j = tid >> 1;
            int col = 0, len = 0;
            if (j < ns) {
              int bp, bq;
              rr_pair(rank + (c0 + j) * nctas, r, nb, bp, bq);
              const int b = (tid & 1) ? bq : bp;
              col = (int)((int64_t)K * b / nb);
              len = (int)((int64_t)K * (b + 1) / nb) - col;
            }
            s_col32[tid] = col;
            s_len32[tid] = len;
          }
          __syncthreads();
          // one bulk copy per column (ld is even: every column starts 16-byte aligned and is
          // ld FP32 complex long, a multiple of 16 bytes; the staging stride is ld too)
          if (tid == 0) {
            uint32_t bytes = 0;
            for (int j = 0; j < 2 * ns; ++j) bytes += (uint32_t)s_len32[j] * (uint32_t)ld * 8u;
            fence_to_async();
            stage_expect(&s_bar32, bytes + (stall ? 16u : 0u));
            for (int j = 0; j < 2 * ns; ++j)
              for (int c = 0; c < s_len32[j]; ++c)
                bulk_load(sm + ((int64_t)j * bsmax + c) * ld, F + (int64_t)(s_col32[j] + c) * ld, (uint32_t)ld * 8u,
                          &s_bar32);
          }
          for (int j = 0; j < 2 * ns; ++j)
            for (int c = tid; c < s_len32[j]; c += blockDim.x) smn[j * bsmax + c] = __ldcg(nrm + s_col32[j] + c);
          dead = __syncthreads_or(!stage_wait(&s_bar32, stage_parity, stall));
          if (dead) break;
          stage_parity ^= 1u;
          if (r == 0) {
            const int mpb = bsmax + (bsmax & 1);
            const int P = 2 * ns * (mpb / 2);
            const int G = group_width32(2 * ns_ref * (mpb / 2), R, nwarps), per = 32 / G, slot = warp * per + lane / G;
            for (int rr = 0; rr < mpb - 1; ++rr) {
              for (int base = 0; base < P; base += nwarps * per) {
                const int k = base + slot, j = k / (mpb / 2);
                int a = 0, b = 0;
                bool valid = k < P;
                if (valid) {
                  rr_pair(k % (mpb / 2), rr, mpb, a, b);
                  valid = a < s_len32[j] && b < s_len32[j];
                }
                rot |= jacobi_pair32(sm, R, Rr, ld, smn, j * bsmax + min(a, b), j * bsmax + max(a, b), valid, G,
                                     tol, floor2);
              }
              __syncthreads();
            }
          }
          {
            const int P = ns * bsmax;
            const int G = group_width32(ns_ref * bsmax, R, nwarps), per = 32 / G, slot = warp * per + lane / G;
            for (int t = 0; t < bsmax; ++t) {
              for (int base = 0; base < P; base += nwarps * per) {
                const int k = base + slot, j = k / bsmax, i = k % bsmax;
                int p = 0, q = 0;
                bool valid = false;
                if (k < P) {
                  const int la = s_len32[2 * j], lb = s_len32[2 * j + 1];
                  const bool swap = la > lb;
                  const int sa = swap ? lb : la, sb = swap ? la : lb;
                  valid = i < sa && t < sb;
                  if (valid) {
                    const int pa = (2 * j + (swap ? 1 : 0)) * bsmax + i;
                    const int pb = (2 * j + (swap ? 0 : 1)) * bsmax + (i + t) % sb;
                    p = min(pa, pb);
                    q = max(pa, pb);
                  }
                }
                rot |= jacobi_pair32(sm, R, Rr, ld, smn, p, q, valid, G, tol, floor2);
              }
              if (t + 1 == bsmax) fence_stage();
              __syncthreads();
            }
          }
          if (tid == 0) {
            for (int j = 0; j < 2 * ns; ++j)
              for (int c = 0; c < s_len32[j]; ++c)
                bulk_store(F + (int64_t)(s_col32[j] + c) * ld, sm + ((int64_t)j * bsmax + c) * ld, (uint32_t)ld * 8u);
            bulk_store_drain();
          }
          for (int j = 0; j < 2 * ns; ++j)
            for (int c = tid; c < s_len32[j]; c += blockDim.x) __stcg(nrm + s_col32[j] + c, smn[j * bsmax + c]);
          __syncthreads();
        }
        sync();
      }
      if (rot) s_rot32 = 1;
      __syncthreads();
      if (tid == 0 && s_rot32) __stcg(flags + sweep, 1);
      if (tid == 0 && dead) __stcg(flags + max_sweeps, 1);
      sync();
      converged = __ldcg(flags + sweep) == 0;
      if (__ldcg(flags + max_sweeps) != 0) {
        if (dead) stage_wait(&s_bar32, stage_parity, stall);
        return kSvdExpired;
      }
    }
    return sweep;
  }
};
struct NoJacobi32 {};
struct FrontStart {};      // no FP32 sweeps: a refined sector's front has run them

// S.vd holds ns columns V of K (ld K), unitary to about 1e-5: one Cholesky QR makes V unitary (V^dag V = U^dag U,
// V <- V U^-1), and S.a1 (column c at S.a1 + c * jld) becomes J V in its first ns columns, zero in the rest.  Every
// CTA of the cluster calls it.
template <class Sync>
__device__ void orthonormal_start(const SvdSector& S, const Work& w, const double2* J, int jlen, int jld, int K, int ns,
                                  int rank, int nctas, Sync sync, int max_sweeps) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarps = blockDim.x >> 5;
  const int tid_all = rank * blockDim.x + tid, threads_all = nctas * blockDim.x;
  const int worker = rank * nwarps + warp, workers = nctas * nwarps;
  double2* Vd = S.vd;     // K x ns, column-major (ld K)
  double2* G = S.gm;      // ns x ns, column-major
  // Gram matrix G = Vd^dag Vd (upper triangle; a warp per entry)
  for (int64_t e = worker; e < (int64_t)ns * ns; e += workers) {
    const int a = (int)(e % ns), b = (int)(e / ns);
    if (a > b) continue;
    const double2* va = Vd + (int64_t)a * K;
    const double2* vb = Vd + (int64_t)b * K;
    double gr = 0.0, gi = 0.0;
    for (int k = lane; k < K; k += 32) {
      const double2 x = L2Mem::ld(va + k), y = L2Mem::ld(vb + k);
      gr = fma(x.x, y.x, fma(x.y, y.y, gr));      // conj(x) y
      gi = fma(x.x, y.y, fma(-x.y, y.x, gi));
    }
    gr = warp_sum(gr);
    gi = warp_sum(gi);
    if (lane == 0) L2Mem::st(G + (int64_t)b * ns + a, make_double2(gr, gi));
  }
  sync();
  // Cholesky G = U^dag U in place (upper triangle), column by column
  for (int j = 0; j < ns; ++j) {
    if (tid_all == 0) {
      const double2 gjj = L2Mem::ld(G + (int64_t)j * ns + j);
      L2Mem::st(G + (int64_t)j * ns + j, make_double2(sqrt(fmax(gjj.x, 1e-300)), 0.0));
    }
    sync();
    const double d = L2Mem::ld(G + (int64_t)j * ns + j).x, id = 1.0 / d;
    for (int c = j + 1 + tid_all; c < ns; c += threads_all) {   // row j of U
      const double2 x = L2Mem::ld(G + (int64_t)c * ns + j);
      L2Mem::st(G + (int64_t)c * ns + j, make_double2(x.x * id, x.y * id));
    }
    sync();
    // trailing update G[a, c] -= conj(U[j, a]) U[j, c], j < a <= c
    const int tr = ns - j - 1;
    for (int64_t e = tid_all; e < (int64_t)tr * tr; e += threads_all) {
      const int a = j + 1 + (int)(e % tr), c = j + 1 + (int)(e / tr);
      if (a > c) continue;
      const double2 ua = L2Mem::ld(G + (int64_t)a * ns + j), uc = L2Mem::ld(G + (int64_t)c * ns + j);
      double2 x = L2Mem::ld(G + (int64_t)c * ns + a);
      x.x -= ua.x * uc.x + ua.y * uc.y;
      x.y -= ua.x * uc.y - ua.y * uc.x;
      L2Mem::st(G + (int64_t)c * ns + a, x);
    }
    sync();
  }
  // V <- Vd U^-1, row by row (x U = v by forward substitution; a warp per row)
  for (int k = worker; k < K; k += workers) {
    for (int c = 0; c < ns; ++c) {
      double sr = 0.0, si = 0.0;
      for (int a = lane; a < c; a += 32) {
        const double2 x = L2Mem::ld(Vd + (int64_t)a * K + k), u = L2Mem::ld(G + (int64_t)c * ns + a);
        sr = fma(x.x, u.x, fma(-x.y, u.y, sr));
        si = fma(x.x, u.y, fma(x.y, u.x, si));
      }
      sr = warp_sum(sr);
      si = warp_sum(si);
      if (lane == 0) {
        const double2 v = L2Mem::ld(Vd + (int64_t)c * K + k);
        const double id = 1.0 / L2Mem::ld(G + (int64_t)c * ns + c).x;
        L2Mem::st(Vd + (int64_t)c * K + k, make_double2((v.x - sr) * id, (v.y - si) * id));
      }
      __syncwarp();
    }
  }
  sync();
  // A1 = J V (jlen x ns), the remaining columns zero
  double2* A1 = S.a1;
  for (int64_t e = tid_all; e < (int64_t)K * jlen; e += threads_all) {
    const int t = (int)(e / jlen), i = (int)(e % jlen);
    double ar = 0.0, ai = 0.0;
    if (t < ns) {
      const double2* vt = Vd + (int64_t)t * K;
      for (int k = 0; k < K; ++k) {
        const double2 x = L2Mem::ld(J + (int64_t)k * jld + i), v = L2Mem::ld(vt + k);
        ar = fma(x.x, v.x, fma(-x.y, v.y, ar));
        ai = fma(x.x, v.y, fma(x.y, v.x, ai));
      }
    }
    L2Mem::st(A1 + (int64_t)t * jld + i, make_double2(ar, ai));
  }
  for (int s = tid_all; s <= max_sweeps; s += threads_all) L2Mem::st(w.flags + s, 0);
  sync();
}

// The mixed-precision start of a cluster sector's sweeps (see above).  J: jlen x K, column c at
// J + c * jld (FP64, L2).  On return the FP64 Jacobi matrix is S.a1 (same jld), its first
// *nsel_out columns J V and the rest zero.  Every CTA of the cluster calls it.  False when a
// wait expired (in every CTA alike).
template <class Sync>
__device__ bool mixed_precondition(const SvdSector& S, const Work& w, const double2* J, int jlen, int jld, int K,
                                   int rank, int nctas, Sync sync, double floor2, int max_sweeps,
                                   const JacobiBlocks32& j32, int* nsel_out) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarps = blockDim.x >> 5;
  const int tid_all = rank * blockDim.x + tid, threads_all = nctas * blockDim.x;
  const int worker = rank * nwarps + warp, workers = nctas * nwarps;
  const int Rr = jlen + K, fld = (Rr + 1) & ~1;   // even: columns 16-byte aligned for bulk copies
  float2* F = S.f32;
  // scale so that the largest column has norm 1 (keeps the FP32 squares far from underflow)
  double cmax = 0.0;
  for (int j = 0; j < K; ++j) cmax = fmax(cmax, L2Mem::ld(w.nrm + j));
  const double sc = cmax > 0.0 ? 1.0 / sqrt(cmax) : 1.0;
  for (int64_t e = tid_all; e < (int64_t)K * Rr; e += threads_all) {
    const int c = (int)(e / Rr), i = (int)(e % Rr);
    float2 v = make_float2(0.f, 0.f);
    if (i < jlen) {
      const double2 x = L2Mem::ld(J + (int64_t)c * jld + i);
      v = make_float2((float)(x.x * sc), (float)(x.y * sc));
    } else if (i - jlen == c) {
      v.x = 1.f;
    }
    __stcg(F + (int64_t)c * fld + i, v);
  }
  for (int s = tid_all; s <= max_sweeps; s += threads_all) L2Mem::st(w.flags + s, 0);
  sync();
  // FP32 sweeps to FP32 convergence; the floor is a tenth of the FP64 one (in the scaled units)
  const float tol32 = 1.1920929e-07f * (float)max(jlen, 32);
  const float fl32 = (float)(0.01 * floor2 * sc * sc);
  bool conv32 = false;
  if (j32(F, jlen, Rr, fld, K, S.nrm32, w.flags, rank, nctas, sync, tol32, fl32, min(max_sweeps, S.fp32_sweeps),
          conv32) == kSvdExpired)
    return false;
  for (int j = worker; j < K; j += workers) {   // final FP32 norms
    const float2* a = F + (int64_t)j * fld;
    float acc = 0.f;
    for (int i = lane; i < jlen; i += 32) {
      const float2 x = __ldcg(a + i);
      acc = fmaf(x.x, x.x, fmaf(x.y, x.y, acc));
    }
    acc = warp_sum_f(acc);
    if (lane == 0) __stcg(S.nrm32 + j, acc);
  }
  sync();
  if (tid_all == 0) {   // the kept columns, in column order
    int ns = 0;
    for (int c = 0; c < K; ++c)
      if (__ldcg(S.nrm32 + c) > fl32) __stcg(S.sel + ns++, c);
    __stcg(S.sel + K, ns);
  }
  sync();
  const int ns = __ldcg(S.sel + K);
  for (int64_t e = tid_all; e < (int64_t)K * ns; e += threads_all) {
    const int t = (int)(e / K), k = (int)(e % K);
    const float2 v = __ldcg(F + (int64_t)__ldcg(S.sel + t) * fld + jlen + k);
    L2Mem::st(S.vd + e, make_double2((double)v.x, (double)v.y));
  }
  sync();
  orthonormal_start(S, w, J, jlen, jld, K, ns, rank, nctas, sync, max_sweeps);
  *nsel_out = ns;
  return true;
}

// ---------------------------------------------------------------------------------------
// Front of the refined SVD of a sector (one cluster): M's columns in order of decreasing norm,
// Householder QR, J = R^dag, FP32 one-sided Jacobi on J accumulating the rotations V.  The
// refinement of k_refine.cu then makes J V orthogonal to FP64 rounding on the tensor cores.
//
// QR: the columns are sorted once and not pivoted again; on the lambda-graded sectors that costs
// at most one more FP32 sweep than pivoting at every step (7 -> 8 on evolved and synthetic
// sectors of 51-197 columns), and a column step needs one cluster barrier instead of five: the
// warp that owns column k + 1 applies reflector k to it first and forms reflector k + 1 before
// it goes on with its other columns.
// ---------------------------------------------------------------------------------------

// Column-major Householder QR of K reflectors over ncol columns (column j at A + pos(j) * ld) by all
// warps of the cluster; a column belongs to one warp.  u_k stays in rows k.. of column k, R_kk goes
// to rkk[k], 2 / u^dag u to tau[k].  ush: the CTA's copy of u_k (rows complex).
template <typename T2> struct RealOf;
template <> struct RealOf<double2> { using type = double; };
template <> struct RealOf<float2> { using type = float; };
__device__ __forceinline__ double real_sqrt(double x) { return sqrt(x); }
__device__ __forceinline__ float real_sqrt(float x) { return sqrtf(x); }
__device__ __forceinline__ double warp_sum_t(double v) { return warp_sum(v); }
__device__ __forceinline__ float warp_sum_t(float v) {
#pragma unroll
  for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
template <typename T2, class Pos, class Sync>
__device__ void qr_columns(T2* A, int64_t ld, int rows, int ncol, int K, T2* rkk, typename RealOf<T2>::type* tau,
                           Pos pos, T2* ush, int rank, int nctas, Sync sync) {
  using T = typename RealOf<T2>::type;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarps = blockDim.x >> 5;
  const int worker = rank * nwarps + warp, workers = nctas * nwarps;
  auto reflector = [&](int k) {      // one warp: column k is final above row k
    T2* x = A + (int64_t)pos(k) * ld;
    T s0 = 0, s1 = 0;
    for (int i = k + lane; i < rows; i += 32) {
      const T2 v = x[i];
      s0 = fma(v.x, v.x, s0);
      s1 = fma(v.y, v.y, s1);
    }
    const T x2 = warp_sum_t(s0 + s1);
    const T xn = real_sqrt(x2);
    const T2 x0 = x[k];
    const T a0 = real_sqrt(x0.x * x0.x + x0.y * x0.y);
    T2 beta;
    if (a0 > 0) {
      const T f = -xn / a0;
      beta.x = x0.x * f;
      beta.y = x0.y * f;
    } else {
      beta.x = -xn;
      beta.y = 0;
    }
    const T uu = 2 * x2 + 2 * xn * a0;
    __syncwarp();
    if (lane == 0) {
      T2 u0;
      u0.x = x0.x - beta.x;
      u0.y = x0.y - beta.y;
      x[k] = u0;
      __stcg(rkk + k, beta);
      __stcg(tau + k, uu > 0 ? 2 / uu : T(0));
    }
    __syncwarp();
  };
  if (worker == 0) reflector(0);
  for (int k = 0; k < K; ++k) {
    sync();
    const T2* xk = A + (int64_t)pos(k) * ld;
    const T tk = __ldcg(tau + k);
    for (int i = k + tid; i < rows; i += blockDim.x) ush[i] = __ldcg(xk + i);
    __syncthreads();
    // columns j = worker (mod workers) beyond k, the next one first
    int j0 = worker + (k + 1 - worker + workers - 1) / workers * workers;
    if (k + 1 <= worker) j0 = worker;
    for (int j = j0; j < ncol; j += 2 * workers) {
      const bool two = j + workers < ncol;
      T2* xa = A + (int64_t)pos(j) * ld;
      T2* xb = A + (int64_t)pos(two ? j + workers : j) * ld;
      T pa = 0, qa = 0, pb = 0, qb = 0, ra = 0, sa = 0, rb = 0, sb = 0;
      for (int i = k + lane; i < rows; i += 32) {
        const T2 u = ush[i], a = xa[i], b = xb[i];
        pa = fma(u.x, a.x, pa);
        ra = fma(u.y, a.y, ra);
        qa = fma(u.x, a.y, qa);
        sa = fma(-u.y, a.x, sa);
        pb = fma(u.x, b.x, pb);
        rb = fma(u.y, b.y, rb);
        qb = fma(u.x, b.y, qb);
        sb = fma(-u.y, b.x, sb);
      }
      pa += ra;
      qa += sa;
      pb += rb;
      qb += sb;
#pragma unroll
      for (int o = 16; o; o >>= 1) {
        pa += __shfl_xor_sync(0xffffffffu, pa, o);
        qa += __shfl_xor_sync(0xffffffffu, qa, o);
        pb += __shfl_xor_sync(0xffffffffu, pb, o);
        qb += __shfl_xor_sync(0xffffffffu, qb, o);
      }
      pa *= tk;
      qa *= tk;
      pb *= tk;
      qb *= tk;
      for (int i = k + lane; i < rows; i += 32) {
        const T2 u = ush[i];
        T2 a = xa[i];
        a.x = fma(-u.x, pa, fma(u.y, qa, a.x));
        a.y = fma(-u.x, qa, fma(-u.y, pa, a.y));
        xa[i] = a;
        if (two) {
          T2 b = xb[i];
          b.x = fma(-u.x, pb, fma(u.y, qb, b.x));
          b.y = fma(-u.x, qb, fma(-u.y, pb, b.y));
          xb[i] = b;
        }
      }
      __syncwarp();
      if (j == k + 1 && k + 1 < K) reflector(k + 1);
    }
  }
  sync();
}

// FP32 block-Jacobi sweeps of a front: the K columns of F (column c at F + c * ld, its rows in pairs) in
// 2 cl g blocks, paired by the round-robin order, CTA `rank` at its positions rank g .. rank g + g - 1.  Between
// two rounds every position passes its blocks on to its neighbours, so of the 2 g blocks that a CTA holds it
// keeps all but two in shared memory: it stores those to F and, past the cluster barrier, loads the two that
// arrive.  A CTA whose shared memory holds only gs < g pairs goes through them gs at a time.
// A block pair's shorter block is held in registers, E row pairs a lane of the G lanes of a slot, and meets
// the columns of the other (G = 0: columns too long for that, both in memory).
// A round's exchange takes some 6 us (stores 2.5, the barrier and its slowest CTA 2, loads 1.5), a step 1-1.7 us.
// With every block staged in every round and (re, im) columns read and written for each rotation, a layer at
// chi = 333 (L = 33) took 32.1 ms and one at chi = 512 (L = 32) 86.9, now 28.6 and 73.6.
struct FrontBlocks {
  float2* sm;
  float* smn;
  int bsmax, g, gs, cl;
  int* left;      // set when a bounded wait expires: the sector then goes to the FP64 sweeps
  bool stall;     // expect bytes that no copy brings

  struct Tables {      // one per CTA
    int held[2 * kMaxStaged];      // the block in each slot (-1: none)
    int col[2 * kMaxStaged], len[2 * kMaxStaged];
    int at[2 * kMaxStaged];        // the slot of each block of the stage: pair j's at 2 j and 2 j + 1
    int fresh[2 * kMaxStaged];     // the slot was loaded for this stage
    int swap[kMaxStaged];          // pair j's shorter block is the second
    int most;                      // columns of the stage's longest block
    int dead;                      // a wait of this CTA expired: it holds no columns any more
    uint64_t bar;
  };

  // Makes the slots hold the blocks of stage (r, c0), or none with r < 0; barrier(): between stores and loads.
  template <class Barrier>
  __device__ __forceinline__ void stage(Tables& T, float2* F, int ld, int K, float* nrm, int rank, int r, int c0,
                                        uint32_t& parity, Barrier barrier) const {
    const int tid = threadIdx.x, lane = tid & 31, nb = 2 * cl * g, slots = 2 * gs;
    fence_stage();
    __syncthreads();
    if (T.dead) {
      barrier();
      return;
    }
    int to = -1, want = -1, col = 0, len = 0;
    if (tid < 32) {
      const int held = lane < slots ? T.held[lane] : -1, j = lane >> 1;
      if (r >= 0 && lane < slots && c0 + j < g) {
        int bp, bq;
        rr_pair(rank * g + c0 + j, r, nb, bp, bq);
        want = lane & 1 ? bq : bp;
        col = (int)((int64_t)K * want / nb);
        len = (int)((int64_t)K * (want + 1) / nb) - col;
      }
      bool stays = false;
      for (int s = 0; s < slots; ++s) {
        if (__shfl_sync(0xffffffffu, held, s) == want && want >= 0) to = s;
        if (__shfl_sync(0xffffffffu, want, s) == held && held >= 0) stays = true;
      }
      if (held >= 0 && !stays) {
        const int from = T.col[lane], n = T.len[lane];
        for (int c = 0; c < n; ++c) {
          bulk_store(F + (int64_t)(from + c) * ld, sm + (lane * bsmax + c) * ld, (uint32_t)ld * 8u);
          __stcg(nrm + from + c, smn[lane * bsmax + c]);
        }
      }
      bulk_store_drain();
      unsigned room = __ballot_sync(0xffffffffu, lane < slots && !stays);
      const bool load = want >= 0 && to < 0;
      const unsigned loads = __ballot_sync(0xffffffffu, load);
      for (int i = __popc(loads & ((1u << lane) - 1)); i; --i) room &= room - 1;
      if (load) to = __ffs(room) - 1;
      __syncwarp();
      if (lane < slots) {
        T.fresh[lane] = 0;
        if (!stays) T.held[lane] = -1;
      }
      __syncwarp();
      if (want >= 0) {
        T.at[lane] = to;
        T.held[to] = want;
        T.col[to] = col;
        T.len[to] = len;
        T.fresh[to] = load;
      }
      const int other = __shfl_xor_sync(0xffffffffu, len, 1);
      if (want >= 0 && !(lane & 1)) T.swap[j] = len > other;
      const int most = __reduce_max_sync(0xffffffffu, len);
      if (lane == 0) T.most = most;
      __syncwarp();
    }
    barrier();
    if (r < 0) return;
    if (tid < 32) {
      const bool load = want >= 0 && T.fresh[to];
      int bytes = load ? len * ld * 8 : 0;
#pragma unroll
      for (int o = 16; o; o >>= 1) bytes += __shfl_xor_sync(0xffffffffu, bytes, o);
      fence_to_async();
      if (lane == 0) stage_expect(&T.bar, (uint32_t)bytes + (stall ? 16u : 0u));
      __syncwarp();
      if (load)
        for (int c = 0; c < len; ++c)
          bulk_load(sm + (to * bsmax + c) * ld, F + (int64_t)(col + c) * ld, (uint32_t)ld * 8u, &T.bar);
    }
    for (int e = tid; e < slots * bsmax; e += blockDim.x) {
      const int s = e / bsmax, c = e % bsmax;
      if (T.held[s] >= 0 && T.fresh[s] && c < T.len[s]) smn[e] = __ldcg(nrm + T.col[s] + c);
    }
    if (__syncthreads_or(!stage_wait(&T.bar, parity, stall))) {
      if (tid < slots) {
        T.at[tid] = tid;
        T.len[tid] = 0;
      }
      if (tid == 0) {
        *left = T.dead = 1;
        T.most = 0;
      }
      __syncthreads();
      return;
    }
    parity ^= 1u;
  }

  template <int G, int E, class Sync>
  __device__ void sweeps(Tables& T, float2* F, int R2, int Rr2, int ld, int K, float* nrm, int* flags, int rank,
                         Sync sync, float tol, float floor2, int max_sweeps) const {
    const int tid = threadIdx.x, warp = tid >> 5, nwarps = blockDim.x >> 5;
    const int ring = 2 * cl * g - 1;
    uint32_t parity = 0;
    if (tid == 0) {
      stage_bar_init(&T.bar);
      T.dead = 0;
    }
    if (tid < 2 * gs) T.held[tid] = -1;
    __syncthreads();
    stage(T, F, ld, K, nrm, rank, 0, 0, parity, [] { __syncthreads(); });
    for (int sweep = 0;; ++sweep) {
      bool far = false;
      for (int r = 0; r < ring; ++r)
        for (int c0 = 0; c0 < g; c0 += gs) {
          const int ns = min(gs, g - c0);
          if (r == 0) {      // fresh norms, and the pairs inside each block
            for (int e = warp; e < 2 * ns * bsmax; e += nwarps) {
              const int s = T.at[e / bsmax], c = e % bsmax;
              if (c < T.len[s]) norm32(sm + (s * bsmax + c) * ld, R2, smn + s * bsmax + c);
            }
            __syncthreads();
            const int mpb = bsmax + (bsmax & 1), P = 2 * ns * (mpb / 2);
            const int W = group_width32(P, 2 * R2, nwarps), slots = blockDim.x / W;
            for (int rr = 0; rr < mpb - 1; ++rr) {
              for (int k0 = 0; k0 < P; k0 += slots) {
                const int k = k0 + tid / W;
                int a = 0, b = 0, s = 0;
                bool valid = k < P;
                if (valid) {
                  s = T.at[k / (mpb / 2)];
                  rr_pair(k % (mpb / 2), rr, mpb, a, b);
                  valid = a < T.len[s] && b < T.len[s];
                }
                far |= pair32(sm, R2, Rr2, ld, smn, s * bsmax + min(a, b), s * bsmax + max(a, b), valid, W, tol,
                              floor2) > kFp32Stop * kFp32Stop;
              }
              __syncthreads();
            }
          }
          const int most = T.most, P = ns * most;
          if constexpr (G > 0) {
            constexpr int slots = kBlockThreads / G;
            for (int k0 = 0; k0 < P; k0 += slots) {
              const int k = k0 + tid / G, j = k / most, i = k % most;
              int own = 0, base = 0, sb = 0;
              bool on = k < P;
              if (on) {
                const int sa = T.at[2 * j + T.swap[j]], so = T.at[2 * j + 1 - T.swap[j]];
                own = sa * bsmax + i;
                base = so * bsmax;
                sb = T.len[so];
                on = i < T.len[sa];
              }
              Held32<G, E> x;
              if (on) x.load(sm + own * ld, Rr2, smn[own]);
              int c = i;      // it meets base + (i + t) mod sb
              for (int t = 0; t < most; ++t) {
                const bool live = on && t < sb;
                const int q = live ? base + c : 0;
                if (++c >= sb) c = 0;
                far |= x.meet(sm + q * ld, smn + q, R2, Rr2, live, tol, floor2) > kFp32Stop * kFp32Stop;
                __syncthreads();
              }
              if (on) {
                x.store(sm + own * ld, Rr2);
                if ((tid & (G - 1)) == 0) smn[own] = x.al;
              }
            }
          } else {
            const int W = group_width32(P, 2 * R2, nwarps), slots = blockDim.x / W;
            for (int t = 0; t < most; ++t) {
              for (int k0 = 0; k0 < P; k0 += slots) {
                const int k = k0 + tid / W, j = k / most, i = k % most;
                int p = 0, q = 0;
                bool valid = k < P;
                if (valid) {
                  const int sa = T.at[2 * j + T.swap[j]], so = T.at[2 * j + 1 - T.swap[j]];
                  valid = i < T.len[sa] && t < T.len[so];
                  if (valid) {
                    p = sa * bsmax + i;
                    q = so * bsmax + (i + t) % T.len[so];
                  }
                }
                far |= pair32(sm, R2, Rr2, ld, smn, p, q, valid, W, tol, floor2) > kFp32Stop * kFp32Stop;
              }
              __syncthreads();
            }
          }
          const bool over = c0 + gs >= g, last = over && r + 1 == ring;
          if (!last) {
            if (over) stage(T, F, ld, K, nrm, rank, r + 1, 0, parity, sync);
            else stage(T, F, ld, K, nrm, rank, r, c0 + gs, parity, [] { __syncthreads(); });
          }
        }
      if (__syncthreads_or(far) && tid == 0) __stcg(flags + sweep, 1);
      if (tid == 0 && T.dead) __stcg(flags + max_sweeps, 1);
      bool done = false;
      stage(T, F, ld, K, nrm, rank, 0, 0, parity, [&] {
        sync();
        done = __ldcg(flags + sweep) == 0 || sweep + 1 >= max_sweeps || __ldcg(flags + max_sweeps) != 0;
      });
      if (done) break;
    }
    stage(T, F, ld, K, nrm, rank, -1, 0, parity, sync);
    if (T.dead) stage_wait(&T.bar, parity, stall);
  }

  template <class Sync>
  __device__ void operator()(float2* F, int R2, int Rr2, int ld, int K, float* nrm, int* flags, int rank, Sync sync,
                             float tol, float floor2, int max_sweeps) const {
    __shared__ Tables T;
    if (max_sweeps < 1) return;
    if (Rr2 <= 192) sweeps<16, 12>(T, F, R2, Rr2, ld, K, nrm, flags, rank, sync, tol, floor2, max_sweeps);
    else if (Rr2 <= 256) sweeps<32, 8>(T, F, R2, Rr2, ld, K, nrm, flags, rank, sync, tol, floor2, max_sweeps);
    else if (Rr2 <= 384) sweeps<32, 12>(T, F, R2, Rr2, ld, K, nrm, flags, rank, sync, tol, floor2, max_sweeps);
    else sweeps<0, 0>(T, F, R2, Rr2, ld, K, nrm, flags, rank, sync, tol, floor2, max_sweeps);
  }
};

template <class Sync>
__device__ void svd_front(const SvdSector& S, const Work& w, int rank, int nctas, Sync sync, int max_sweeps,
                          const FrontBlocks& j32, unsigned char* smem) {
  const int m = S.m, n = S.n, K = min(m, n);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarps = blockDim.x >> 5;
  const int tid_all = rank * blockDim.x + tid, threads_all = nctas * blockDim.x;
  const int worker = rank * nwarps + warp, workers = nctas * nwarps;
  double2* W = w.W;            // column-major, m rows
  // ---- M = diag(lambda) Theta', transposed to columns: a warp moves 4 rows x 8 columns ----
  {
    const int tr = (m + 3) / 4, tc = (n + 7) / 8;
    for (int64_t t = worker; t < (int64_t)tr * tc; t += workers) {
      const int i = (int)(t / tc) * 4 + (lane >> 3), j = (int)(t % tc) * 8 + (lane & 7);
      if (i < m && j < n) {
        const double s = S.rowscale ? S.rowscale[i] : 1.0;
        const double2 x = S.theta[(int64_t)i * n + j];
        __stcg(W + (int64_t)j * m + i, make_double2(s * x.x, s * x.y));
      }
    }
  }
  if (tid_all < 16) __stcg(S.rstate + tid_all, 0);
  sync();
  for (int j = worker; j < n; j += workers) {
    double a0 = 0.0, a1 = 0.0;
    for (int i = lane; i < m; i += 32) {
      const double2 x = __ldcg(W + (int64_t)j * m + i);
      a0 = fma(x.x, x.x, a0);
      a1 = fma(x.y, x.y, a1);
    }
    a0 = warp_sum(a0 + a1);
    if (lane == 0) __stcg(w.nu + j, a0);
  }
  sync();
  // descending order of the column norms (NaN last: the order stays a permutation), |M|_F^2
  double fro2 = 0.0;
  for (int j = lane; j < n; j += 32) fro2 += __ldcg(w.nu + j);
  fro2 = warp_sum(fro2);
  for (int j = tid_all; j < n; j += threads_all) {
    const double vj = __ldcg(w.nu + j), v = isnan(vj) ? -1.0 : vj;
    int rk = 0;
    for (int q = 0; q < n; ++q) {
      const double wq = __ldcg(w.nu + q), x = isnan(wq) ? -1.0 : wq;
      rk += (x > v) || (x == v && q < j);
    }
    __stcg(w.perm + rk, j);
  }
  if (!(fro2 > 1e-270 && fro2 < 1e270)) {      // zero, not finite, or squares out of range
    if (tid_all == 0) __stcg(S.rstate + 1, 1);
    return;
  }
  const int sc = -(ilogb(fro2) / 2);            // J is scaled so that |J|_F is about 1 (exactly, by 2^sc)
  const double scale = scalbn(1.0, sc);
  const double frel = fmax(32.0 * kEps, S.floor_rel);
  const double floor2 = fmax(frel * frel * fro2, S.floor_abs * S.floor_abs) * scale * scale;
  if (tid_all == 0) {
    S.rfloor2[0] = floor2;
    S.rfloor2[1] = scalbn(1.0, -sc);
  }
  sync();
  const int* perm = w.perm;
  qr_columns(W, (int64_t)m, m, n, K, w.u, w.nu0, [&](int j) { return __ldcg(perm + j); },
             reinterpret_cast<double2*>(smem), rank, nctas, sync);

  // ---- J = R^dag: column i (n long) is the conjugate of row i of R, in sorted column order ----
  double2* J = S.J;
  const bool wide = S.wide;
  const int jlen = wide ? K : n;
  const int vr = even32(jlen), fld = vr + even32(K);      // the rotations' first row, the columns' stride
  float2* F = S.F;
  float2* F1 = reinterpret_cast<float2*>(S.A1);     // wide: FP32 J, n x K, for a second QR
  {
    const int tr = (K + 3) / 4, tc = (n + 7) / 8;
    for (int64_t t = worker; t < (int64_t)tr * tc; t += workers) {
      const int i = (int)(t / tc) * 4 + (lane & 3), j = (int)(t % tc) * 8 + (lane >> 2);
      if (i < K && j < n) {
        double2 x = make_double2(0.0, 0.0);
        if (i == j) x = __ldcg(w.u + i);
        else if (i < j) x = __ldcg(W + (int64_t)__ldcg(perm + j) * m + i);
        x.x *= scale;
        x.y *= -scale;
        J[(int64_t)i * n + j] = x;
        const float2 f = make_float2((float)x.x, (float)x.y);
        if (wide) __stcg(F1 + (int64_t)i * n + j, f);
        else set_row32(F + (int64_t)i * fld, j, f);
      }
    }
  }
  for (int s = tid_all; s <= max_sweeps; s += threads_all) L2Mem::st(w.flags + s, 0);
  if (wide) {      // FP32 QR of J: the sweeps rotate the K x K factor, the rotations are the same
    sync();
    float2* rk = reinterpret_cast<float2*>(w.u);      // m >= K entries
    float* tk = reinterpret_cast<float*>(w.nu0);
    qr_columns(F1, (int64_t)n, n, K, K, rk, tk, [](int j) { return j; }, reinterpret_cast<float2*>(smem), rank, nctas,
               sync);
    for (int64_t e = tid_all; e < (int64_t)K * K; e += threads_all) {
      const int c = (int)(e / K), i = (int)(e % K);
      float2 v = make_float2(0.f, 0.f);
      if (i == c) v = __ldcg(rk + c);
      else if (i < c) v = __ldcg(F1 + (int64_t)c * n + i);
      set_row32(F + (int64_t)c * fld, i, v);
    }
  }
  for (int64_t e = tid_all; e < (int64_t)K * (fld - jlen); e += threads_all) {   // V = I below
    const int c = (int)(e / (fld - jlen)), i = jlen + (int)(e % (fld - jlen));
    set_row32(F + (int64_t)c * fld, i, make_float2(i - vr == c ? 1.f : 0.f, 0.f));
  }
  sync();
  // ---- FP32 sweeps to FP32 convergence; the floor is a tenth of the FP64 one -------------------
  fence_stage();      // the staging area held reflectors
  __syncthreads();
  const float tol32 = 1.1920929e-07f * (float)max(jlen, 32);
  const float fl32 = (float)(0.01 * floor2);
  j32(F, vr / 2, fld / 2, fld, K, S.nrm32, w.flags, rank, sync, tol32, fl32, min(max_sweeps, S.fp32_sweeps + 6));
  for (int j = worker; j < K; j += workers) {   // final FP32 norms, past what L1 holds of the columns
    const float2* a = F + (int64_t)j * fld;
    float acc = 0.f;
    for (int i = lane; i < vr; i += 32) {
      const float2 x = __ldcg(a + i);
      acc = fmaf(x.x, x.x, fmaf(x.y, x.y, acc));
    }
    acc = warp_sum_f(acc);
    if (lane == 0) __stcg(S.nrm32 + j, acc);
  }
  sync();
  if (tid_all < 32) {   // the kept columns, in column order
    int ns = 0;
    for (int c0 = 0; c0 < K; c0 += 32) {
      const bool keep = c0 + lane < K && __ldcg(S.nrm32 + c0 + lane) > fl32;
      const unsigned mask = __ballot_sync(0xffffffffu, keep);
      if (keep) __stcg(S.sel + ns + __popc(mask & ((1u << lane) - 1)), c0 + lane);
      ns += __popc(mask);
    }
    if (lane == 0) {
      __stcg(S.rstate, ns);
      if (ns == 0) __stcg(S.rstate + 1, 1);
    }
  }
  sync();
  const int ns = __ldcg(S.rstate);
  for (int64_t e = tid_all; e < (int64_t)K * ns; e += threads_all) {
    const int t = (int)(e / K), k = (int)(e % K);
    const float* v = reinterpret_cast<const float*>(F + (int64_t)__ldcg(S.sel + t) * fld + vr + (k & ~1)) + (k & 1);
    S.V0[e] = make_double2((double)__ldcg(v), (double)__ldcg(v + 2));
  }
  sync();      // F is read
  float2* V32 = S.V32();
  for (int64_t e = tid_all; e < (int64_t)K * ns; e += threads_all) V32[e] = make_float2((float)S.V0[e].x, (float)S.V0[e].y);
}

template <class Mem, class Sync, class Jacobi, class J32 = NoJacobi32>
__device__ void svd_sector(const SvdSector& S, const Work& w, int rank, int nctas, Sync sync, int max_sweeps,
                           Jacobi jacobi, J32 j32 = J32()) {
  __shared__ double red_d[kMaxWarps][33];
  __shared__ double red_v[kMaxWarps];
  __shared__ int red_i[kMaxWarps];
  const int m = S.m, n = S.n, K = min(m, n), ld = odd_ld(n);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarps = blockDim.x >> 5;
  const int tid_all = rank * blockDim.x + tid, threads_all = nctas * blockDim.x;
  const int worker = rank * nwarps + warp, workers = nctas * nwarps;
  double2* W = w.W;
  // A sector whose refinement did not settle (large groups of close values) goes on from the front's J and rotations: no
  // second QR, no second FP32 sweeps.  300 x 300 with its values in equal pairs: 147 -> 78 ms.
  // Compiled for the kernel that follows the refinement alone: in the others the branch cost QR and sweeps (one update
  // at chi = 2048 in TF32 on a team: 166 ms without, 186 with it).
  bool resume = false;
  if constexpr (std::is_same<J32, FrontStart>::value) resume = __ldcg(S.rstate + 1) >= kLeftAt;
  if (resume) {
    const double up = S.rfloor2[1];      // J is scaled
    for (int64_t e = tid_all; e < (int64_t)K * n; e += threads_all) {
      const double2 x = S.J[e];
      Mem::st(W + e / n * ld + e % n, make_double2(up * x.x, up * x.y));
    }
    for (int s = tid_all; s <= max_sweeps; s += threads_all) Mem::st(w.flags + s, 0);
    sync();
    for (int j = worker; j < K; j += workers) {
      double acc = 0.0;
      for (int i = lane; i < n; i += 32) {
        const double2 x = Mem::ld(W + (int64_t)j * ld + i);
        acc = fma(x.x, x.x, fma(x.y, x.y, acc));
      }
      acc = warp_sum(acc);
      if (lane == 0) Mem::st(w.nu + j, acc);
    }
    sync();
    if (tid_all == 0) {
      double f = 0.0;
      for (int j = 0; j < K; ++j) f += Mem::ld(w.nu + j);
      Mem::st(w.scal + 1, f);
    }
    sync();
  } else {
    // ---- load M = diag(lambda) Theta' (row-major), column norms, identity permutation ----
    const int64_t mn = (int64_t)m * n;
    for (int64_t e = tid_all; e < mn; e += threads_all) {
      const int i = (int)(e / n), j = (int)(e % n);
      const double s = S.rowscale ? S.rowscale[i] : 1.0;
      const double2 t = S.theta[e];
      Mem::st(W + (int64_t)i * ld + j, make_double2(s * t.x, s * t.y));
    }
    for (int s = tid_all; s <= max_sweeps; s += threads_all) Mem::st(w.flags + s, 0);
    sync();
    for (int j = tid_all; j < n; j += threads_all) {
      double acc = 0.0;
      for (int i = 0; i < m; ++i) {
        const double2 x = Mem::ld(W + (int64_t)i * ld + j);
        acc = fma(x.x, x.x, fma(x.y, x.y, acc));
      }
      Mem::st(w.nu + j, acc);
      Mem::st(w.nu0 + j, acc);
      Mem::st(w.perm + j, j);
    }
    sync();
    if (tid_all == 0) {
      double f = 0.0;
      for (int j = 0; j < n; ++j) f += Mem::ld(w.nu + j);
      Mem::st(w.scal + 1, f);
    }
    sync();

    // ---- Householder QR with column pivoting: M P = Q R ---------------------------------
    for (int k = 0; k < K; ++k) {
      // pivot: largest remaining partial norm, ties to the smaller index
      double bv = -1.0;
      int bi = n;
      for (int j = k + tid_all; j < n; j += threads_all) {
        const double v = Mem::ld(w.nu + j);
        if (v > bv || (v == bv && j < bi)) { bv = v; bi = j; }
      }
#pragma unroll
      for (int o = 16; o; o >>= 1) {
        const double ov = __shfl_xor_sync(0xffffffffu, bv, o);
        const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
        if (ov > bv || (ov == bv && oi < bi)) { bv = ov; bi = oi; }
      }
      if (lane == 0) { red_v[warp] = bv; red_i[warp] = bi; }
      __syncthreads();
      if (tid == 0) {
        for (int x = 1; x < nwarps; ++x)
          if (red_v[x] > bv || (red_v[x] == bv && red_i[x] < bi)) { bv = red_v[x]; bi = red_i[x]; }
        Mem::st(w.pv + rank, bv);
        Mem::st(w.pi + rank, bi);
      }
      sync();
      if (nctas <= kMaxCluster) {
        bv = Mem::ld(w.pv);
        bi = Mem::ld(w.pi);
        for (int x = 1; x < nctas; ++x) {
          const double v = Mem::ld(w.pv + x);
          const int ix = Mem::ld(w.pi + x);
          if (v > bv || (v == bv && ix < bi)) { bv = v; bi = ix; }
        }
      } else {
        bv = -1.0;
        bi = n;
        for (int x = lane; x < nctas; x += 32) {
          const double v = Mem::ld(w.pv + x);
          const int ix = Mem::ld(w.pi + x);
          if (v > bv || (v == bv && ix < bi)) { bv = v; bi = ix; }
        }
#pragma unroll
        for (int o = 16; o; o >>= 1) {
          const double ov = __shfl_xor_sync(0xffffffffu, bv, o);
          const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
          if (ov > bv || (ov == bv && oi < bi)) { bv = ov; bi = oi; }
        }
      }
      const int p = (bi < n) ? bi : k;
      if (p != k) {
        for (int i = tid_all; i < m; i += threads_all) {
          double2* rowp = W + (int64_t)i * ld;
          const double2 a = Mem::ld(rowp + k), b = Mem::ld(rowp + p);
          Mem::st(rowp + k, b);
          Mem::st(rowp + p, a);
        }
        if (tid_all == 0) {
          double a = Mem::ld(w.nu + k), b = Mem::ld(w.nu + p);
          Mem::st(w.nu + k, b); Mem::st(w.nu + p, a);
          a = Mem::ld(w.nu0 + k); b = Mem::ld(w.nu0 + p);
          Mem::st(w.nu0 + k, b); Mem::st(w.nu0 + p, a);
          const int ia = Mem::ld(w.perm + k), ib = Mem::ld(w.perm + p);
          Mem::st(w.perm + k, ib); Mem::st(w.perm + p, ia);
        }
      }
      sync();
      // reflector H = I - (2 / u^dag u) u u^dag with H x = beta e_k, |beta| = |x|
      if (worker == 0) {
        double x2 = 0.0;
        for (int i = k + lane; i < m; i += 32) {
          const double2 x = Mem::ld(W + (int64_t)i * ld + k);
          x2 = fma(x.x, x.x, fma(x.y, x.y, x2));
        }
        x2 = warp_sum(x2);
        const double xn = sqrt(x2);
        const double2 x0 = Mem::ld(W + (int64_t)k * ld + k);
        const double a0 = hypot(x0.x, x0.y);
        double2 beta;
        if (a0 > 0.0) beta = make_double2(-x0.x / a0 * xn, -x0.y / a0 * xn);
        else beta = make_double2(-xn, 0.0);
        const double uu = 2.0 * x2 + 2.0 * xn * a0;
        for (int i = k + lane; i < m; i += 32) {
          double2 x = Mem::ld(W + (int64_t)i * ld + k);
          if (i == k) x = make_double2(x.x - beta.x, x.y - beta.y);
          Mem::st(w.u + i, x);
          Mem::st(W + (int64_t)i * ld + k, i == k ? beta : make_double2(0.0, 0.0));
        }
        if (lane == 0) Mem::st(w.scal, uu > 0.0 ? 2.0 / uu : 0.0);
      }
      sync();
      // trailing update W[k:, j] -= (2/u^dag u) u (u^dag W[k:, j]) for j > k: a CTA takes tiles of tc columns,
      // each column's dot product in nwarps interleaved row chunks (summed in order whatever the tile
      // width).  32 columns fill the CTA's warps; with more CTAs than such tiles narrower ones put the
      // chunks of several columns into a warp, so that every CTA has FP64 work.
      constexpr int ahead = Mem::kCache ? kAhead : 1;      // shared memory answers at once
      const double sc = Mem::ld(w.scal);
      const int ncols = n - k - 1;
      int tc = 32;
      if constexpr (Mem::kCache)
        while (nctas > kMaxCluster && tc > 8 && (ncols + tc / 2 - 1) / (tc / 2) <= nctas) tc >>= 1;
      const int ntiles = (ncols + tc - 1) / tc;
      const int tcol = tid % tc, chunk = tid / tc;      // chunks beyond nwarps have no rows in the dot product
      if (sc != 0.0) {
        for (int tile = rank; tile < ntiles; tile += nctas) {
          const int j = k + 1 + tile * tc + tcol;
          double pr = 0.0, pim = 0.0;
          if (j < n && chunk < nwarps) {
#pragma unroll ahead
            for (int i = k + chunk; i < m; i += nwarps) {
              const double2 ui = Mem::ld(w.u + i);
              const double2 x = Mem::ld(W + (int64_t)i * ld + j);
              pr = fma(ui.x, x.x, fma(ui.y, x.y, pr));      // conj(u_i) x
              pim = fma(ui.x, x.y, fma(-ui.y, x.x, pim));
            }
          }
          if (chunk < nwarps) red_d[chunk][tcol] = pr;
          __syncthreads();
          double wr = 0.0;
          for (int x = 0; x < nwarps; ++x) wr += red_d[x][tcol];
          __syncthreads();
          if (chunk < nwarps) red_d[chunk][tcol] = pim;
          __syncthreads();
          double wi = 0.0;
          for (int x = 0; x < nwarps; ++x) wi += red_d[x][tcol];
          __syncthreads();
          wr *= sc;
          wi *= sc;
          if (j < n) {
            const int step = (int)blockDim.x / tc;
            for (int i0 = k + chunk; i0 < m; i0 += ahead * step) {
              double2 ui[ahead], x[ahead];
#pragma unroll
              for (int a = 0; a < ahead; ++a)
                if (i0 + a * step < m) {
                  ui[a] = Mem::ld(w.u + i0 + a * step);
                  x[a] = Mem::ld(W + (int64_t)(i0 + a * step) * ld + j);
                }
#pragma unroll
              for (int a = 0; a < ahead; ++a)
                if (i0 + a * step < m) {
                  x[a].x -= ui[a].x * wr - ui[a].y * wi;
                  x[a].y -= ui[a].x * wi + ui[a].y * wr;
                  Mem::st(W + (int64_t)(i0 + a * step) * ld + j, x[a]);
                }
            }
          }
          __syncthreads();
          if (chunk == 0 && j < n) {       // downdate the partial norm, recompute on cancellation
            const double2 r = Mem::ld(W + (int64_t)k * ld + j);
            double v = Mem::ld(w.nu + j) - (r.x * r.x + r.y * r.y);
            if (v <= 1.4901161193847656e-8 * Mem::ld(w.nu0 + j)) {
              v = 0.0;
              for (int i = k + 1; i < m; ++i) {
                const double2 x = Mem::ld(W + (int64_t)i * ld + j);
                v = fma(x.x, x.x, fma(x.y, x.y, v));
              }
              Mem::st(w.nu0 + j, v);
            }
            Mem::st(w.nu + j, v);
          }
        }
      } else {
        for (int tile = rank; tile < ntiles; tile += nctas) {
          const int j = k + 1 + tile * tc + tcol;
          if (chunk == 0 && j < n) {
            const double2 r = Mem::ld(W + (int64_t)k * ld + j);
            Mem::st(w.nu + j, fmax(Mem::ld(w.nu + j) - (r.x * r.x + r.y * r.y), 0.0));
          }
        }
      }
      sync();
    }

    // ---- R^dag: conjugate rows 0..K-1 in place; they are the Jacobi columns ------------
    for (int64_t e = tid_all; e < (int64_t)K * n; e += threads_all) {
      const int i = (int)(e / n), j = (int)(e % n);
      double2* a = W + (int64_t)i * ld + j;
      const double2 x = Mem::ld(a);
      Mem::st(a, make_double2(x.x, -x.y));
    }
    sync();
  }
  const double fro2 = Mem::ld(w.scal + 1);

  // ---- wide sectors (K = m < n): R^dag = Q2 [R2; 0] by unpivoted Householder QR of its
  // K columns.  Rotations that orthogonalise the columns of R^dag orthogonalise those of
  // R2 alike (Q2 has orthonormal columns), so the Jacobi sweeps run on R2's columns,
  // length K instead of n, and Y = P Q2 [normalised columns; 0] at the end. --------------
  double2* J = W;        // the Jacobi matrix: column j at J + j * jld, length jlen
  int jlen = n, jld = ld;
  double* tau = w.nu;    // reflector scales (w.nu is free after the pivoted QR; n >= K)
  const bool wide = Mem::kCache && S.wide;   // cluster kernels only (their scratch holds R2)
  if constexpr (Mem::kCache) if (wide) {
    double2* W2 = S.work2;
    const int ld2 = odd_ld(K);
    for (int64_t e = tid_all; e < (int64_t)K * ld2; e += threads_all) Mem::st(W2 + e, make_double2(0.0, 0.0));
    sync();
    for (int k = 0; k < K; ++k) {
      double2* xk = W + (int64_t)k * ld;
      if (worker == 0) {   // H_k = I - tau_k v v^dag maps x_k[k:] to beta e_k; v overwrites x_k[k:]
        double x2 = 0.0;
        for (int i = k + lane; i < n; i += 32) {
          const double2 x = Mem::ld(xk + i);
          x2 = fma(x.x, x.x, fma(x.y, x.y, x2));
        }
        x2 = warp_sum(x2);
        const double xn = sqrt(x2);
        const double2 x0 = Mem::ld(xk + k);
        const double a0 = hypot(x0.x, x0.y);
        double2 beta;
        if (a0 > 0.0) beta = make_double2(-x0.x / a0 * xn, -x0.y / a0 * xn);
        else beta = make_double2(-xn, 0.0);
        const double uu = 2.0 * x2 + 2.0 * xn * a0;
        if (lane == 0) {
          Mem::st(xk + k, make_double2(x0.x - beta.x, x0.y - beta.y));
          Mem::st(tau + k, uu > 0.0 ? 2.0 / uu : 0.0);
          Mem::st(W2 + (int64_t)k * ld2 + k, beta);          // R2[k][k]
        }
      }
      sync();
      const double tk = Mem::ld(tau + k);
      for (int j = k + 1 + worker; j < K; j += workers) {
        double2* xj = W + (int64_t)j * ld;
        double pr = 0.0, pim = 0.0;
        if (tk != 0.0) {
          for (int i = k + lane; i < n; i += 32) {
            const double2 v = Mem::ld(xk + i), x = Mem::ld(xj + i);
            pr = fma(v.x, x.x, fma(v.y, x.y, pr));         // conj(v) x
            pim = fma(v.x, x.y, fma(-v.y, x.x, pim));
          }
          pr = warp_sum(pr) * tk;
          pim = warp_sum(pim) * tk;
        }
        for (int i = k + lane; i < n; i += 32) {
          double2 x = Mem::ld(xj + i);
          if (tk != 0.0) {
            const double2 v = Mem::ld(xk + i);
            x.x -= v.x * pr - v.y * pim;
            x.y -= v.x * pim + v.y * pr;
            Mem::st(xj + i, x);
          }
          if (i == k) Mem::st(W2 + (int64_t)j * ld2 + k, x);   // R2[k][j], final after H_k
        }
      }
      sync();
    }
    J = W2;
    jlen = K;
    jld = ld2;
  }
  for (int j = worker; j < K; j += workers) {
    const double2* a = J + (int64_t)j * jld;
    double acc = 0.0;
    for (int i = lane; i < jlen; i += 32) {
      const double2 x = Mem::ld(a + i);
      acc = fma(x.x, x.x, fma(x.y, x.y, acc));
    }
    acc = warp_sum(acc);
    if (lane == 0) Mem::st(w.nrm + j, acc);
  }
  sync();

  // ---- one-sided Jacobi on the K columns of R^dag (or R2) --------------------------------
  const double tol = kEps * (double)max(n, 32);
  const double tol2 = tol * tol;
  // floor: the rounding-noise level 32 eps |M|_F, or the caller's deflation level when higher
  const double frel = fmax(32.0 * kEps, S.floor_rel);
  const double floor2 = fmax(frel * frel * fro2, S.floor_abs * S.floor_abs);
  bool converged = false;
  int Kj = K;                    // columns the FP64 sweeps rotate
  bool start = resume;
  if constexpr (std::is_same<J32, JacobiBlocks32>::value) start = S.f32 && K >= 2;
  if constexpr (!std::is_same<J32, NoJacobi32>::value) {
    if (start) {       // the FP64 sweeps start from J V, V the rotations of FP32 sweeps
      int ns = K;
      if constexpr (std::is_same<J32, FrontStart>::value) {
        ns = __ldcg(S.rstate);
        const float2* V32 = S.V32();
        for (int64_t e = tid_all; e < (int64_t)K * ns; e += threads_all)
          Mem::st(S.vd + e, make_double2((double)V32[e].x, (double)V32[e].y));
        sync();
        orthonormal_start(S, w, J, jlen, jld, K, ns, rank, nctas, sync, max_sweeps);
      } else if (!mixed_precondition(S, w, J, jlen, jld, K, rank, nctas, sync, floor2, max_sweeps, j32, &ns)) {
        if (tid_all == 0) *S.status = kSvdExpired;
        return;
      }
      J = S.a1;
      Kj = ns;
      for (int j = worker; j < K; j += workers) {   // column norms of the new Jacobi matrix
        const double2* a = J + (int64_t)j * jld;
        double acc = 0.0;
        for (int i = lane; i < jlen; i += 32) {
          const double2 x = Mem::ld(a + i);
          acc = fma(x.x, x.x, fma(x.y, x.y, acc));
        }
        acc = warp_sum(acc);
        if (lane == 0) Mem::st(w.nrm + j, acc);
      }
      sync();
    }
  }
  const int sweep = jacobi(J, jlen, jld, Kj, w, rank, nctas, sync, tol2, floor2, max_sweeps, converged);
  if (sweep == kSvdExpired) {
    if (tid_all == 0) *S.status = kSvdExpired;
    return;
  }

  // ---- singular values (noise floor -> 0), descending, ties by column index -----------
  for (int j = worker; j < K; j += workers) {
    const double2* a = J + (int64_t)j * jld;
    double acc = 0.0;
    for (int i = lane; i < jlen; i += 32) {
      const double2 x = Mem::ld(a + i);
      acc = fma(x.x, x.x, fma(x.y, x.y, acc));
    }
    acc = warp_sum(acc);
    if (lane == 0) Mem::st(w.nrm + j, acc <= floor2 ? 0.0 : sqrt(acc));
  }
  sync();
  for (int j = tid_all; j < K; j += threads_all) {
    const double vj = Mem::ld(w.nrm + j);
    const double v = isnan(vj) ? -1.0 : vj;       // NaN ranks last: ranks stay a permutation
    int rk = 0;
    for (int q = 0; q < K; ++q) {
      const double wq = Mem::ld(w.nrm + q);
      const double x = isnan(wq) ? -1.0 : wq;
      rk += (x > v) || (x == v && q < j);
    }
    Mem::st(w.ord + rk, j);
  }
  sync();
  for (int r = tid_all; r < K; r += threads_all) S.sigma[r] = Mem::ld(w.nrm + Mem::ld(w.ord + r));
  if (wide) {
    // Y[perm[j], r] = (Q2 [R2 column ord[r] / sigma_r; 0])[j]; Q2 = H_0 ... H_{K-1}, one warp per column
    for (int r = worker; r < K; r += workers) {
      const int c = Mem::ld(w.ord + r);
      const double sv = Mem::ld(w.nrm + c);
      double2* y = S.ytmp + (int64_t)r * n;
      if (sv > 0.0) {
        const double2* a = J + (int64_t)c * jld;
        for (int i = lane; i < n; i += 32) {
          double2 val = make_double2(0.0, 0.0);
          if (i < K) {
            const double2 x = Mem::ld(a + i);
            val = make_double2(x.x / sv, x.y / sv);
          }
          Mem::st(y + i, val);
        }
        __syncwarp();
        for (int k = K - 1; k >= 0; --k) {
          const double tk = Mem::ld(tau + k);
          if (tk == 0.0) continue;
          const double2* v = W + (int64_t)k * ld;
          double pr = 0.0, pim = 0.0;
          for (int i = k + lane; i < n; i += 32) {
            const double2 vv = Mem::ld(v + i), x = Mem::ld(y + i);
            pr = fma(vv.x, x.x, fma(vv.y, x.y, pr));
            pim = fma(vv.x, x.y, fma(-vv.y, x.x, pim));
          }
          pr = warp_sum(pr) * tk;
          pim = warp_sum(pim) * tk;
          for (int i = k + lane; i < n; i += 32) {
            const double2 vv = Mem::ld(v + i);
            double2 x = Mem::ld(y + i);
            x.x -= vv.x * pr - vv.y * pim;
            x.y -= vv.x * pim + vv.y * pr;
            Mem::st(y + i, x);
          }
          __syncwarp();
        }
        for (int j = lane; j < n; j += 32) S.Y[(int64_t)r * n + Mem::ld(w.perm + j)] = Mem::ld(y + j);
      } else {
        for (int j = lane; j < n; j += 32) S.Y[(int64_t)r * n + j] = make_double2(0.0, 0.0);
      }
    }
  } else {
    // Y[perm[j], r] = column ord[r] of R^dag, row j, divided by its norm
    for (int64_t e = tid_all; e < (int64_t)K * n; e += threads_all) {
      const int r = (int)(e / n), j = (int)(e % n);
      const int c = Mem::ld(w.ord + r);
      const double sv = Mem::ld(w.nrm + c);
      double2 y = make_double2(0.0, 0.0);
      if (sv > 0.0) {
        const double2 a = Mem::ld(J + (int64_t)c * jld + j);
        y = make_double2(a.x / sv, a.y / sv);
      }
      S.Y[(int64_t)r * n + Mem::ld(w.perm + j)] = y;
    }
  }
  if (tid_all == 0) {
    *S.status = converged ? sweep : -1;
    if (S.path) *S.path = MPS_SVD_SWEEPS | (start ? MPS_SVD_FP32_START : 0) | Sync::kPath | Jacobi::kPath;
  }
}

struct CtaSync {
  static constexpr int kPath = 0;
  __device__ void operator()() const { __syncthreads(); }
};
struct ClusterSync {
  static constexpr int kPath = 0;
  __device__ void operator()() const { cluster_sync_all(); }
};

// The barrier of a team: CTAs of one cooperative launch (all resident) that share a sector.  bar[0] counts
// arrivals, zero at the launch.  The wait is bounded (about 20 s): a CTA whose wait expires marks the
// sector and leaves; no bulk copy is in flight at a barrier, so nothing outlives it.
struct TeamSync {
  static constexpr int kPath = MPS_SVD_TEAM;
  unsigned* bar;
  int* status;
  unsigned size;
  unsigned* target;      // shared memory, thread 0's: arrivals that complete the present barrier
  __device__ void operator()() const {
    __shared__ int s_expired;
    __syncthreads();
    if (threadIdx.x == 0) {
      int expired = 0;
      *target += size;
      asm volatile("fence.acq_rel.gpu;\n" ::: "memory");
      atomicAdd(bar, 1u);
      const long long t0 = clock64();
      for (;;) {
        unsigned v;
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];\n" : "=r"(v) : "l"(bar) : "memory");
        if ((int)(v - *target) >= 0) break;
        if (clock64() - t0 > 40000000000LL) {
          expired = 1;
          break;
        }
      }
      asm volatile("fence.acq_rel.gpu;\n" ::: "memory");
      s_expired = expired;
      if (expired) *status = kSvdExpired;
    }
    __syncthreads();
    if (s_expired) asm volatile("exit;\n");
  }
};

// shared-memory layout of the one-CTA kernel (offsets in bytes)
struct SmemLayout {
  int64_t W, u, nu, nu0, perm, nrm, ord, flags, pv, pi, scal, total;
};
__host__ __device__ inline SmemLayout smem_layout(int m, int n) {
  auto al = [](int64_t x) { return (x + 15) & ~int64_t(15); };
  const int K = m < n ? m : n;
  SmemLayout L;
  int64_t o = 0;
  L.W = o; o = al(o + 16LL * m * odd_ld(n));
  L.u = o; o = al(o + 16LL * m);
  L.nu = o; o = al(o + 8LL * n);
  L.nu0 = o; o = al(o + 8LL * n);
  L.perm = o; o = al(o + 4LL * n);
  L.nrm = o; o = al(o + 8LL * K);
  L.ord = o; o = al(o + 4LL * K);
  L.flags = o; o = al(o + 4LL * (kJacobiMaxSweeps + 1));
  L.pv = o; o = al(o + 8);
  L.pi = o; o = al(o + 4);
  L.scal = o; o = al(o + 16);
  L.total = o;
  return L;
}

__device__ __forceinline__ void cta_sector(const SvdSector& S, unsigned char* smem_raw, int max_sweeps) {
  const SmemLayout L = smem_layout(S.m, S.n);
  Work w;
  w.W = reinterpret_cast<double2*>(smem_raw + L.W);
  w.u = reinterpret_cast<double2*>(smem_raw + L.u);
  w.nu = reinterpret_cast<double*>(smem_raw + L.nu);
  w.nu0 = reinterpret_cast<double*>(smem_raw + L.nu0);
  w.perm = reinterpret_cast<int*>(smem_raw + L.perm);
  w.nrm = reinterpret_cast<double*>(smem_raw + L.nrm);
  w.ord = reinterpret_cast<int*>(smem_raw + L.ord);
  w.flags = reinterpret_cast<int*>(smem_raw + L.flags);
  w.pv = reinterpret_cast<double*>(smem_raw + L.pv);
  w.pi = reinterpret_cast<int*>(smem_raw + L.pi);
  w.scal = reinterpret_cast<double*>(smem_raw + L.scal);
  svd_sector<PlainMem>(S, w, 0, 1, CtaSync{}, max_sweeps, JacobiRoundRobin<PlainMem>{});
}

__global__ void __launch_bounds__(kSvdThreads, 1) jacobi_cta_kernel(const SvdSector* __restrict__ secs,
                                                                    int max_sweeps) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cta_sector(secs[blockIdx.x], smem_raw, max_sweeps);
}

// ---------------------------------------------------------------------------------------
// One CTA, everything in shared memory: the refined SVD of a small sector.  The QR and the FP32 sweeps are
// those of svd_front; up to kSmallK columns the refinement runs here too (its products are shorter than a
// kernel launch), above that J and V go to the tensor-core kernels.  The FP64 sweeps of jacobi_cta_kernel
// paid for every rotation's root and quotient in FP64 (some 1500 cycles of latency a pair); here those
// are FP32 and the FP64 work is the QR and the refinement's products.  A front of 95 x 95 takes 2.07 ms, 0.84
// of it the QR (0.6 at the SM's FP64 rate), 1.17 the FP32 sweeps; on a cluster of 8 over L2 it took 3.3.  A whole 15 x 15
// sector takes 116 us, 39 in the QR, 28 in the sweeps, 42 in two refinement steps: chains of FP64 roots, quotients
// and sums.
// ---------------------------------------------------------------------------------------
struct SmallLayout {
  int ldm, fld, lda;                  // strides of W, F and A
  int64_t W, F, V, V32, E, rkk, tau, nu, lam, inv, nrm, perm, sel, rank, total;
};
__host__ __device__ inline SmallLayout small_layout(int m, int n, bool full) {
  auto al = [](int64_t x) { return (x + 15) & ~int64_t(15); };
  const int K = m < n ? m : n;
  SmallLayout L;
  L.ldm = m | 1;
  L.fld = even32(n) + even32(K);
  L.lda = n | 1;
  int64_t o = 0;
  const int64_t w = 16LL * L.ldm * n, f = 8LL * L.fld * K, a = 16LL * L.lda * K;
  L.W = o;
  if (full) {      // A takes F's place
    o = al(o + w);
    L.F = o; o = al(o + (f > a ? f : a));
  } else {         // J goes to global memory, then F takes W's place
    L.F = o; o = al(o + (f > w ? f : w));
  }
  L.V = o; o = al(o + (full ? 16LL * K * K : 0));
  L.V32 = o; o = al(o + (full ? 8LL * K * K : 0));
  L.E = o; o = al(o + (full ? 8LL * K * K : 0));
  L.rkk = o; o = al(o + 16LL * K);
  L.tau = o; o = al(o + 8LL * K);
  L.nu = o; o = al(o + 8LL * n);
  L.lam = o; o = al(o + 8LL * K);
  L.inv = o; o = al(o + 8LL * K);
  L.nrm = o; o = al(o + 4LL * K);
  L.perm = o; o = al(o + 4LL * n);
  L.sel = o; o = al(o + 4LL * K);
  L.rank = o; o = al(o + 4LL * K);
  L.total = o;
  return L;
}

// Householder QR of a matrix in shared memory by one CTA (as qr_columns).  An FP64 instruction occupies its
// quarter of the SM for 64 cycles whatever its lanes do, so a step's chain of them is its time: warp 0
// takes column k + 1 with all its lanes on the rows and forms the next reflector (its two roots are one
// instruction sequence on two lanes), while the other warps share the rest, 8, 4 or 2 columns a warp with
// the rows dealt to 4, 8 or 16 lanes: no lane idles and the sums end in 2-4 shuffles.  35 x 35 took 248 us
// with a warp per pair of columns, 142 with 8 columns a warp throughout.
template <class Pos>
__device__ void qr_small(double2* A, int ld, int rows, int ncol, int K, double2* rkk, double* tau, Pos pos) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarps = blockDim.x >> 5;
  // column j <- (I - tau_k u u^dag) column j by the lanes sub, sub + subs, ... that share it
  auto apply = [&](const double2* u, double tk, double2* x, int k, int sub, int subs, bool on) {
    double p = 0.0, q = 0.0, r = 0.0, s = 0.0;
    if (on)
      for (int i = k + sub; i < rows; i += subs) {
        const double2 a = u[i], b = x[i];
        p = fma(a.x, b.x, p);
        r = fma(a.y, b.y, r);
        q = fma(a.x, b.y, q);
        s = fma(a.y, b.x, s);
      }
    p += r;
    q -= s;
    for (int o = 32 / subs; o < 32; o <<= 1) {      // lanes of a column differ in the high bits
      p += __shfl_xor_sync(0xffffffffu, p, o);
      q += __shfl_xor_sync(0xffffffffu, q, o);
    }
    p *= tk;
    q *= tk;
    if (on) {
#pragma unroll 4
      for (int i = k + sub; i < rows; i += subs) {
        const double2 a = u[i];
        double2 b = x[i];
        b.x = fma(-a.x, p, fma(a.y, q, b.x));
        b.y = fma(-a.x, q, fma(-a.y, p, b.y));
        x[i] = b;
      }
    }
  };
  auto reflector = [&](int k) {      // warp 0: column k is final above row k
    double2* x = A + (int64_t)pos(k) * ld;
    double s0 = 0.0, s1 = 0.0;
    for (int i = k + lane; i < rows; i += 32) {
      const double2 v = x[i];
      s0 = fma(v.x, v.x, s0);
      s1 = fma(v.y, v.y, s1);
    }
    const double x2 = warp_sum(s0 + s1);
    const double2 x0 = x[k];
    const double a2 = fma(x0.x, x0.x, x0.y * x0.y);
    const double v = lane == 0 ? x2 : a2, iv = v > 0.0 ? rsqrt(v) : 0.0, sv = v * iv;
    const double xn = __shfl_sync(0xffffffffu, sv, 0), a0 = __shfl_sync(0xffffffffu, sv, 1);
    const double ia = __shfl_sync(0xffffffffu, iv, 1);
    const double f = -ia * xn;
    const double2 beta = a2 > 0.0 ? make_double2(x0.x * f, x0.y * f) : make_double2(-xn, 0.0);
    const double uu = x2 + xn * a0;
    __syncwarp();
    if (lane == 0) {
      x[k] = make_double2(x0.x - beta.x, x0.y - beta.y);
      rkk[k] = beta;
      tau[k] = uu > 0.0 ? 1.0 / uu : 0.0;
    }
    __syncwarp();
  };
  if (warp == 0) reflector(0);
  for (int k = 0; k < K; ++k) {
    __syncthreads();
    const double2* u = A + (int64_t)pos(k) * ld;
    const double tk = tau[k];
    if (warp == 0) {
      if (k + 1 < ncol) apply(u, tk, A + (int64_t)pos(k + 1) * ld, k, lane, 32, true);
      __syncwarp();
      if (k + 1 < K) reflector(k + 1);
    } else {
      const int rest = ncol - k - 2;
      const int cols = rest > 4 * (nwarps - 1) ? 8 : rest > 2 * (nwarps - 1) ? 4 : 2;
      const int col = lane & (cols - 1), sub = lane / cols;
      for (int j0 = k + 2 + (warp - 1) * cols; j0 < ncol; j0 += (nwarps - 1) * cols) {
        const bool on = j0 + col < ncol;
        apply(u, tk, A + (int64_t)pos(on ? j0 + col : k) * ld, k, sub, 32 / cols, on);
      }
    }
  }
  __syncthreads();
}

// FP32 sweeps of one CTA until no pair of a sweep was further than kFp32Stop from orthogonal (each sweep
// squares the distance, so the sweep that found that has left about its square).
//
// Order: the columns are halved, every column of the second half meets every column of the first, then
// each half is treated alike (as many sweeps as the round-robin order, on sectors of 51-197 columns).  The
// Lanes lanes of a slot hold their column of the second half in registers through a level.  Columns longer than
// 2 Lanes E rows, or more of them than slots, go round-robin with both columns in memory (Lanes = 0).
template <int Lanes, int E>
__device__ void small_sweeps(float2* F, int R2, int Rr2, int ld, int K, float* nrm, float tol, float floor2,
                             int max_sweeps) {
  __shared__ int s_far;
  const int tid = threadIdx.x, warp = tid >> 5, nwarps = blockDim.x >> 5;
  for (int sweep = 0; K > 1 && sweep < max_sweeps; ++sweep) {
    for (int j = warp; j < K; j += nwarps) norm32(F + j * ld, R2, nrm + j);
    if (tid == 0) s_far = 0;
    __syncthreads();
    bool far = false;
    if constexpr (Lanes > 0) {
      for (int level = 0; (K - 1) >> level; ++level) {
        // slot u's column: the u-th of the second halves of this level's segments
        int u = tid / Lanes, own = -1, base = 0, len = 0;
        for (int g = 0; g < 1 << level; ++g) {
          int a = 0, b = K;
          for (int k = level - 1; k >= 0; --k) {
            const int h = a + (b - a + 1) / 2;
            if (g >> k & 1) a = h; else b = h;
          }
          const int n2 = (b - a) / 2;
          if (u < n2) {
            base = a;
            len = b - a - n2;
            own = a + len + u;
            break;
          }
          u -= n2;
        }
        const int steps = (((K - 1) >> level) + 2) / 2;      // half of the longest segment, rounded up
        Held32<Lanes, E> x;
        x.load(F + max(own, 0) * ld, Rr2, nrm[max(own, 0)]);
        int c = u;                                           // it meets base + (u + step) mod len
        for (int s = 0; s < steps; ++s) {
          const bool live = own >= 0 && s < len;
          const int q = live ? base + c : 0;
          if (++c >= len) c = 0;
          far |= x.meet(F + q * ld, nrm + q, R2, Rr2, live, tol, floor2) > kFp32Stop * kFp32Stop;
          __syncthreads();
        }
        if (own >= 0) {
          x.store(F + own * ld, Rr2);
          if ((tid & (Lanes - 1)) == 0) nrm[own] = x.al;
        }
        __syncthreads();
      }
    } else {
      const int mp = K + (K & 1), ring = mp - 1, P = mp / 2;
      int G = 8;
      while (G < 32 && 4 * G < Rr2 && 2 * G * P <= (int)blockDim.x) G *= 2;
      const int slots = blockDim.x / G, slot = tid / G;
      for (int r = 0; r < ring; ++r) {
#pragma unroll 1
        for (int k = slot; k < P + slot; k += slots) {      // rr_pair(k, r), the sums being below 2 ring
          const int a = k + r - (k + r >= ring ? ring : 0);
          const int b = k == 0 ? r : ring - k + r - (r >= k ? ring : 0);
          const int p = k == 0 ? 0 : a + 1, q = b + 1;
          const bool valid = k < P && p < K && q < K;
          far |= pair32(F, R2, Rr2, ld, nrm, min(p, q), max(p, q), valid, G, tol, floor2) > kFp32Stop * kFp32Stop;
        }
        __syncthreads();
      }
    }
    if (far) s_far = 1;
    __syncthreads();
    const int go = s_far;
    __syncthreads();
    if (!go) break;
  }
}

// Threads: kSvdThreads for whole refinements (up to kSmallK columns), kFrontThreads for fronts: 4 a column, so
// every pair of a round of up to 96 columns has its 8 lanes.
template <int Threads>
__global__ void __launch_bounds__(Threads, 1) svd_small_kernel(const SvdSector* __restrict__ secs, int max_sweeps) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ int s_ns, s_theta;
  const SvdSector S = secs[blockIdx.x];
  const int m = S.m, n = S.n, K = min(m, n);
  constexpr bool full = Threads == kSvdThreads;      // else the front of a sector that the tensor cores refine
  const SmallLayout L = small_layout(m, n, full);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarps = blockDim.x >> 5;
  double2* W = reinterpret_cast<double2*>(smem_raw + L.W);
  float2* F = reinterpret_cast<float2*>(smem_raw + L.F);
  double2* rkk = reinterpret_cast<double2*>(smem_raw + L.rkk);
  double* tau = reinterpret_cast<double*>(smem_raw + L.tau);
  double* nu = reinterpret_cast<double*>(smem_raw + L.nu);
  float* nrm = reinterpret_cast<float*>(smem_raw + L.nrm);
  int* perm = reinterpret_cast<int*>(smem_raw + L.perm);
  int* sel = reinterpret_cast<int*>(smem_raw + L.sel);
  for (int e = tid; e < m * n; e += blockDim.x) {
    const int i = e / n, j = e % n;
    const double s = S.rowscale ? S.rowscale[i] : 1.0;
    const double2 x = S.theta[e];
    W[(int64_t)j * L.ldm + i] = make_double2(s * x.x, s * x.y);
  }
  if (!full && tid < 16) S.rstate[tid] = 0;
  __syncthreads();
  for (int j = warp; j < n; j += nwarps) {
    double a0 = 0.0, a1 = 0.0;
    for (int i = lane; i < m; i += 32) {
      const double2 x = W[(int64_t)j * L.ldm + i];
      a0 = fma(x.x, x.x, a0);
      a1 = fma(x.y, x.y, a1);
    }
    a0 = warp_sum(a0 + a1);
    if (lane == 0) nu[j] = a0;
  }
  __syncthreads();
  double fro2 = 0.0;
  for (int j = lane; j < n; j += 32) fro2 += nu[j];
  fro2 = warp_sum(fro2);
  for (int j = tid; j < n; j += blockDim.x) {      // descending norms, NaN last
    const double vj = nu[j], v = isnan(vj) ? -1.0 : vj;
    int rk = 0;
    for (int q = 0; q < n; ++q) {
      const double wq = nu[q], x = isnan(wq) ? -1.0 : wq;
      rk += (x > v) || (x == v && q < j);
    }
    perm[rk] = j;
  }
  __syncthreads();
  bool left = !(fro2 > 1e-270 && fro2 < 1e270);      // zero, not finite, or squares out of range
  if (left) {
    if (!full) {
      if (tid == 0) S.rstate[1] = 1;
      return;
    }
  } else {
    const int sc = -(ilogb(fro2) / 2);
    const double scale = scalbn(1.0, sc), up = scalbn(1.0, -sc);
    const double frel = fmax(32.0 * kEps, S.floor_rel);
    const double floor2 = fmax(frel * frel * fro2, S.floor_abs * S.floor_abs) * scale * scale;
    qr_small(W, L.ldm, m, n, K, rkk, tau, [&](int j) { return perm[j]; });
    // R scaled by 2^sc; F = [fl32(R^dag); I]
    if (full) {      // R stays in W, its diagonal in place
      for (int e = tid; e < K * n; e += blockDim.x) {
        const int i = e % K, j = e / K;
        double2* w = W + (int64_t)perm[j] * L.ldm + i;
        double2 x = make_double2(0.0, 0.0);
        if (i <= j) {
          x = i == j ? rkk[i] : *w;
          x.x *= scale;
          x.y *= scale;
          *w = x;
        }
        set_row32(F + i * L.fld, j, make_float2((float)x.x, (float)-x.y));
      }
    } else {         // J = R^dag for the tensor-core kernels
      for (int e = tid; e < K * n; e += blockDim.x) {
        const int i = e / n, j = e % n;
        double2 x = make_double2(0.0, 0.0);
        if (i <= j) x = i == j ? rkk[i] : W[(int64_t)perm[j] * L.ldm + i];
        S.J[e] = make_double2(scale * x.x, -scale * x.y);
      }
      __syncthreads();
      for (int e = tid; e < K * n; e += blockDim.x) {
        const double2 x = S.J[e];
        set_row32(F + e / n * L.fld, e % n, make_float2((float)x.x, (float)x.y));
      }
    }
    const int vr = even32(n);      // the rotations' first row
    for (int e = tid; e < K * (L.fld - n); e += blockDim.x) {
      const int j = e / (L.fld - n), i = n + e % (L.fld - n);
      set_row32(F + j * L.fld, i, make_float2(i - vr == j ? 1.f : 0.f, 0.f));
    }
    __syncthreads();
    const float tol32 = 1.1920929e-07f * (float)max(n, 32), fl32 = (float)(0.01 * floor2);
    const int slots = K / 2, R2 = vr / 2, Rr2 = L.fld / 2, sweeps = min(max_sweeps, S.fp32_sweeps + 6);
    if (full && slots <= Threads / 32 && Rr2 <= 64) small_sweeps<32, 2>(F, R2, Rr2, L.fld, K, nrm, tol32, fl32, sweeps);
    else if (slots <= Threads / 16 && Rr2 <= 48) small_sweeps<16, 3>(F, R2, Rr2, L.fld, K, nrm, tol32, fl32, sweeps);
    else if (slots <= Threads / 16 && Rr2 <= 96) small_sweeps<16, 6>(F, R2, Rr2, L.fld, K, nrm, tol32, fl32, sweeps);
    else if (!full && slots <= Threads / 8 && Rr2 <= 96) small_sweeps<8, 12>(F, R2, Rr2, L.fld, K, nrm, tol32, fl32, sweeps);
    else small_sweeps<0, 0>(F, R2, Rr2, L.fld, K, nrm, tol32, fl32, sweeps);
    for (int j = warp; j < K; j += nwarps) norm32(F + j * L.fld, R2, nrm + j);
    __syncthreads();
    if (warp == 0) {      // the kept columns, in column order
      int ns = 0;
      for (int c0 = 0; c0 < K; c0 += 32) {
        const bool keep = c0 + lane < K && nrm[c0 + lane] > fl32;
        const unsigned mask = __ballot_sync(0xffffffffu, keep);
        if (keep) sel[ns + __popc(mask & ((1u << lane) - 1))] = c0 + lane;
        ns += __popc(mask);
      }
      if (lane == 0) s_ns = ns;
    }
    __syncthreads();
    const int ns = s_ns;
    if (!full) {
      float2* V32 = S.V32();
      for (int e = tid; e < K * ns; e += blockDim.x) {
        const float2 v = row32(F + sel[e / K] * L.fld, vr + e % K);
        S.V0[e] = make_double2((double)v.x, (double)v.y);
        V32[e] = v;
      }
      for (int j = tid; j < n; j += blockDim.x) S.order[j] = perm[j];
      if (tid == 0) {
        S.rfloor2[0] = floor2;
        S.rfloor2[1] = up;
        S.rstate[0] = ns;
        if (ns == 0) S.rstate[1] = 1;
      }
      return;
    }
    // ---- refinement in FP64 (see k_refine.cu) -------------------------------------------------
    double2* V = reinterpret_cast<double2*>(smem_raw + L.V);
    float2* V32 = reinterpret_cast<float2*>(smem_raw + L.V32);
    float2* E = reinterpret_cast<float2*>(smem_raw + L.E);
    double* lam = reinterpret_cast<double*>(smem_raw + L.lam);
    double* inv = reinterpret_cast<double*>(smem_raw + L.inv);
    for (int e = tid; e < K * ns; e += blockDim.x) {
      const float2 v = row32(F + sel[e / K] * L.fld, vr + e % K);
      V32[e] = v;
      V[e] = make_double2((double)v.x, (double)v.y);
    }
    __syncthreads();
    double2* A = reinterpret_cast<double2*>(smem_raw + L.F);
    const float tol = 2.2204460e-16f * (float)max(n, 32);
    int steps = 0;
    bool settled = false;
    left = ns == 0;
    for (int it = 0; !left; ++it) {
      for (int e = tid; e < n * ns; e += blockDim.x) {      // A = J V
        const int j = e % n, c = e / n, top = min(j, K - 1);
        const double2* r = W + (int64_t)perm[j] * L.ldm;
        const double2* v = V + (int64_t)c * K;
        double a0 = 0.0, a1 = 0.0, b0 = 0.0, b1 = 0.0;
        for (int i = 0; i <= top; ++i) {
          a0 = fma(r[i].x, v[i].x, a0);
          a1 = fma(r[i].y, v[i].y, a1);
          b0 = fma(r[i].x, v[i].y, b0);
          b1 = fma(r[i].y, v[i].x, b1);
        }
        A[(int64_t)c * L.lda + j] = make_double2(a0 + a1, b0 - b1);
      }
      __syncthreads();
      for (int c = warp; c < ns; c += nwarps) {
        double a0 = 0.0, a1 = 0.0;
        for (int j = lane; j < n; j += 32) {
          const double2 x = A[(int64_t)c * L.lda + j];
          a0 = fma(x.x, x.x, a0);
          a1 = fma(x.y, x.y, a1);
        }
        a0 = warp_sum(a0 + a1);
        if (lane == 0) {
          lam[c] = a0;
          inv[c] = a0 > 0.0 ? rsqrt(a0) : 0.0;
        }
      }
      if (tid == 0) s_theta = 0;
      __syncthreads();
      if (settled || it == kRefineSteps) break;
      float worst = 0.f;
      for (int e = tid; e < ns * ns; e += blockDim.x) {
        const int p = e % ns, q = e / ns;
        if (p > q) continue;
        const double2 *a = A + (int64_t)p * L.lda, *b = A + (int64_t)q * L.lda, *v = V + (int64_t)p * K,
                      *u = V + (int64_t)q * K;
        double g0 = 0.0, g1 = 0.0, h0 = 0.0, h1 = 0.0;
        for (int i = 0; i < K; ++i) {
          g0 = fma(v[i].x, u[i].x, g0);
          g1 = fma(v[i].y, u[i].y, g1);
          h0 = fma(v[i].x, u[i].y, h0);
          h1 = fma(v[i].y, u[i].x, h1);
        }
        const float rr = (float)((p == q ? 1.0 : 0.0) - (g0 + g1)), ri = (float)(h1 - h0);
        if (p == q) {
          E[q * K + p] = make_float2(0.5f * rr, 0.f);
          worst = fmaxf(worst, fabsf(rr));
          continue;
        }
        g0 = g1 = h0 = h1 = 0.0;
        for (int j = 0; j < n; ++j) {
          g0 = fma(a[j].x, b[j].x, g0);
          g1 = fma(a[j].y, b[j].y, g1);
          h0 = fma(a[j].x, b[j].y, h0);
          h1 = fma(a[j].y, b[j].x, h1);
        }
        RefinePair P = {};
        float rho = 1.f;
        if (fmin(lam[p], lam[q]) > floor2) {
          const double f = inv[p] * inv[q];
          rho = (float)(lam[q] * f);                  // |a_q| / |a_p|
          P = refine_pair(1.f, 1.f, rho, (float)((g0 + g1) * f), (float)((h0 - h1) * f), rr, ri, tol);
          worst = fmaxf(worst, P.size);
        }
        E[q * K + p] = make_float2(P.pq.x * rho, P.pq.y * rho);
        E[p * K + q] = make_float2(P.qp.x / rho, P.qp.y / rho);
        if (!(P.size >= 0.f)) worst = 1e30f;          // NaN: leave it
      }
      for (int o = 16; o; o >>= 1) worst = fmaxf(worst, __shfl_xor_sync(0xffffffffu, worst, o));
      if (lane == 0) atomicMax(&s_theta, __float_as_int(worst));
      __syncthreads();
      const float th = __int_as_float(s_theta);
      left = refine_fails(th, it);
      settled = !left && refine_settles(th, ns, n);
      steps = it + 1;
      if (!left)
        for (int e = tid; e < K * ns; e += blockDim.x) {      // V += V E: E is small, FP32 holds the product
          const int i = e % K, c = e / K;
          float x = 0.f, y = 0.f, sq = 0.f;
          for (int k = 0; k < ns; ++k) {
            const float2 v = V32[k * K + i], w = E[c * K + k];
            sq = fmaf(w.x, w.x, fmaf(w.y, w.y, sq));
            x = fmaf(v.x, w.x, fmaf(-v.y, w.y, x));
            y = fmaf(v.x, w.y, fmaf(v.y, w.x, y));
          }
          const float2 v = V32[e];      // the diagonal's second-order part
          V[e].x += (double)fmaf(-0.5f * sq, v.x, x);
          V[e].y += (double)fmaf(-0.5f * sq, v.y, y);
        }
      __syncthreads();
      for (int e = tid; e < K * ns; e += blockDim.x) V32[e] = make_float2((float)V[e].x, (float)V[e].y);
      __syncthreads();
    }
    if (settled) {      // singular values and Y = P A / sigma in descending order; the rest is zero
      int* rank = reinterpret_cast<int*>(smem_raw + L.rank);
      for (int c = tid; c < K; c += blockDim.x) {
        const double v = c < ns && lam[c] > floor2 ? lam[c] : 0.0;
        int rk = 0;
        for (int j = 0; j < K; ++j) {
          const double x = j < ns && lam[j] > floor2 ? lam[j] : 0.0;
          rk += (x > v) || (x == v && j < c);
        }
        const double sg = sqrt(v);
        S.sigma[rk] = sg * up;
        rank[c] = rk;
        inv[c] = v > 0.0 ? 1.0 / sg : 0.0;
      }
      __syncthreads();
      for (int e = tid; e < n * K; e += blockDim.x) {
        const int j = e % n, c = e / n;
        double2 z = make_double2(0.0, 0.0);
        if (c < ns && inv[c] > 0.0) {
          const double2 a = A[(int64_t)c * L.lda + j];
          z = make_double2(a.x * inv[c], a.y * inv[c]);
        }
        S.Y[(int64_t)rank[c] * n + perm[j]] = z;
      }
      if (tid == 0) {
        *S.status = steps;
        if (S.path) *S.path = MPS_SVD_REFINED;
      }
      return;
    }
  }
  __syncthreads();
  if constexpr (full) cta_sector(S, smem_raw, max_sweeps);      // the FP64 sweeps, from the start
}

__device__ __forceinline__ Work cluster_work(const SvdSector& S) {
  Work w;
  w.W = S.work;
  w.u = S.uwork;
  w.nu = S.norms;
  w.nu0 = S.norms + S.n;
  w.perm = S.order;
  w.nrm = S.norms + 2 * S.n;
  w.ord = S.order + S.n;
  w.flags = S.flags;
  w.pv = S.pivv;
  w.pi = S.flags + kJacobiMaxSweeps + 1;
  w.scal = S.pivv + (S.teambar ? kMaxTeam : kMaxCluster);
  return w;
}

__global__ void __launch_bounds__(kSvdThreads) jacobi_cluster_kernel(const SvdSector* __restrict__ secs,
                                                                     int cluster, int max_sweeps) {
  const int rank = (int)cluster_rank();
  const SvdSector S = secs[blockIdx.x / cluster];
  svd_sector<L2Mem>(S, cluster_work(S), rank, cluster, ClusterSync{}, max_sweeps, JacobiRoundRobin<L2Mem>{});
}

// The block-Jacobi SVD of one sector by nctas CTAs in the ordering of a cluster of cl0; Refined: a sector that has
// passed through a front and the refinement.
template <bool Refined, class Sync>
__device__ __forceinline__ void svd_blocks(const SvdSector& S, unsigned char* smem, int rank, int nctas, int cl0,
                                           Sync sync, int max_sweeps, int stall) {
  const int K = min(S.m, S.n);
  JacobiBlocks jb;
  jb.stall = stall & kStallBlocks;
  jb.g = S.groups;
  jb.gs = S.staged;
  jb.cl0 = cl0;
  jb.bsmax = (K + 2 * cl0 * jb.g - 1) / (2 * cl0 * jb.g);
  jb.sm = reinterpret_cast<double2*>(smem);
  jb.smn = reinterpret_cast<double*>(smem + 16LL * 2 * jb.gs * jb.bsmax * (S.wide ? K : S.n));
  if constexpr (Refined) {
    svd_sector<L2Mem>(S, cluster_work(S), rank, nctas, sync, max_sweeps, jb, FrontStart{});
    return;
  }
  // the FP32 sweeps of a mixed-precision sector stage columns of jlen + K <= 2 jlen FP32
  // complex values in the same area
  JacobiBlocks32 j32;
  j32.stall = jb.stall;
  j32.g = jb.g;
  j32.gs = jb.gs;
  j32.cl0 = cl0;
  j32.bsmax = jb.bsmax;
  j32.sm = reinterpret_cast<float2*>(smem);
  j32.smn = reinterpret_cast<float*>(smem + 8LL * 2 * jb.gs * jb.bsmax * ((((S.wide ? K : S.n) + K) + 1) & ~1));
  svd_sector<L2Mem>(S, cluster_work(S), rank, nctas, sync, max_sweeps, jb, j32);
}

template <bool Refined>
__global__ void __launch_bounds__(kBlockThreads, 2) jacobi_cluster_block_kernel(const SvdSector* __restrict__ secs,
                                                                                int cluster, int max_sweeps, int stall) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const SvdSector S = secs[blockIdx.x / cluster];
  if (Refined && S.rstate[1] == 0 && S.rstate[2] > 0) return;   // settled by the refinement
  svd_blocks<Refined>(S, smem_raw, (int)cluster_rank(), cluster, cluster, ClusterSync{}, max_sweeps, stall);
}

// The same for batches with few large sectors: one cooperative launch, in which a sector has a team
// of S.team_size CTAs (those from S.team_first) instead of a cluster of at most 8.  The block ordering and
// every sum stay those of the cluster, so the results are the same bits; only more SMs share a
// round's block pairs, a column's trailing update and the products.  A chi = 2048 update whose 796 x 796
// sector kept 8 SMs busy for 1.23 s takes 166 ms (a team of 104), three updates at chi = 1024 297 -> 126 ms;
// there the FP64 pipes of the whole chip are the bound.
__global__ void __launch_bounds__(kBlockThreads, 2) jacobi_team_kernel(const SvdSector* __restrict__ secs, int count,
                                                                       int max_sweeps, int stall) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  int k = 0;
  while (k + 1 < count && (int)blockIdx.x >= secs[k + 1].team_first) ++k;
  const SvdSector S = secs[k];
  __shared__ unsigned s_target;
  if (threadIdx.x == 0) s_target = 0;
  svd_blocks<false>(S, smem_raw, (int)blockIdx.x - S.team_first, S.team_size, S.team_cl0,
             TeamSync{S.teambar, S.status, (unsigned)S.team_size, &s_target}, max_sweeps, stall);
}

__global__ void __launch_bounds__(kBlockThreads, 2) svd_front_kernel(const SvdSector* __restrict__ secs, int cluster,
                                                                     int max_sweeps, int stall) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int rank = (int)cluster_rank();
  const SvdSector S = secs[blockIdx.x / cluster];
  const int K = min(S.m, S.n);
  const int fld = even32(S.wide ? K : S.n) + even32(K);
  FrontBlocks j32;
  j32.g = S.groups;
  j32.gs = S.front_staged;
  j32.cl = cluster;
  j32.left = S.rstate + 1;
  j32.stall = stall & kStallFronts;
  j32.bsmax = (K + 2 * cluster * j32.g - 1) / (2 * cluster * j32.g);
  j32.sm = reinterpret_cast<float2*>(smem_raw);
  j32.smn = reinterpret_cast<float*>(smem_raw + 8LL * 2 * j32.gs * j32.bsmax * fld);
  svd_front(S, cluster_work(S), rank, cluster, ClusterSync{}, max_sweeps, j32, smem_raw);
}


}  // namespace

int64_t svd_smem_need(int m, int n) { return smem_layout(m, n).total; }

namespace {

constexpr int kBlockSmemMax = 110 * 1024;   // two block-Jacobi CTAs per SM
constexpr int kFrontSmemMax = 216 * 1024;   // one-CTA fronts
constexpr int kPairSmemMax = 114900;        // cluster fronts, two CTAs per SM
// 8 CTAs per large sector: the GPU places about twice as many 8-CTA clusters as
// 16-CTA ones, which keeps more SMs busy when a layer has hundreds of large sectors
constexpr int kBigCluster = 8;
// Kernel attributes (dynamic shared memory, non-portable clusters) apply to the current device
// only, so they are set once per device, under a lock, with that device's cluster size.
constexpr int kMaxDevices = 64;
std::mutex g_attr_mu;
bool g_attr_done[kMaxDevices] = {};
int g_big_cluster[kMaxDevices] = {};

int64_t block_smem_need(int m, int n, int cl, int g, int gs) {
  const int64_t K = std::min(m, n), bs = (K + 2 * cl * g - 1) / (2 * cl * g);
  return 16 * 2 * gs * bs * n + 16 * 2 * gs * bs + 64;   // norms, and the FP32 staging's even-stride padding
}
// of a front: FP32 columns of at most n + 1 + K + 1 rows, and norms
int64_t front_smem_need(int m, int n, int cl, int g, int gs) {
  const int64_t K = std::min(m, n), bs = (K + 2 * cl * g - 1) / (2 * cl * g);
  return 8 * 2 * gs * bs * (even32(n) + even32((int)K)) + 4 * 2 * gs * bs;
}

cudaError_t set_attrs(int* big_out) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lk(g_attr_mu);
  if (g_attr_done[dev]) {
    *big_out = g_big_cluster[dev];
    return cudaSuccess;
  }
  e = cudaFuncSetAttribute(jacobi_cta_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSvdSmemMax);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(svd_small_kernel<kSvdThreads>, cudaFuncAttributeMaxDynamicSharedMemorySize, kFrontSmemMax);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(svd_small_kernel<kFrontThreads>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             kFrontSmemMax);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(jacobi_cluster_block_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             kBlockSmemMax);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(jacobi_cluster_block_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             kBlockSmemMax);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(svd_front_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kPairSmemMax);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(jacobi_team_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kBlockSmemMax);
  if (e != cudaSuccess) return e;
  // clusters of 16 CTAs are non-portable: use them only where the device can place them
  int big = 8;
  if (cudaFuncSetAttribute(jacobi_cluster_kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) ==
          cudaSuccess &&
      cudaFuncSetAttribute(jacobi_cluster_block_kernel<false>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) ==
          cudaSuccess &&
      cudaFuncSetAttribute(jacobi_cluster_block_kernel<true>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) ==
          cudaSuccess &&
      cudaFuncSetAttribute(svd_front_kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(16);
    cfg.blockDim = dim3(kBlockThreads);
    cfg.dynamicSmemBytes = kBlockSmemMax;
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = 16;
    at.val.clusterDim.y = 1;
    at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, jacobi_cluster_block_kernel<false>, &cfg) == cudaSuccess && n >= 4) big = 16;
  }
  cudaGetLastError();
  g_big_cluster[dev] = big;
  g_attr_done[dev] = true;
  *big_out = big;
  return cudaSuccess;
}

// One cooperative launch of a group of teams.  Two such launches on different streams must not share
// the chip (each could hold SMs that the other's missing CTAs wait for), so every one waits for the
// previous one of its device.
cudaError_t launch_teams(const SvdSector* d, const SvdGroup& g, int max_sweeps, cudaStream_t st) {
  static std::mutex mu;
  static cudaEvent_t last[kMaxDevices] = {};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lk(mu);
  if (!last[dev]) e = cudaEventCreateWithFlags(&last[dev], cudaEventDisableTiming);
  else e = cudaStreamWaitEvent(st, last[dev], 0);
  if (e == cudaSuccess) e = cudaMemsetAsync(g.bar0, 0, (char*)g.bar1 - (char*)g.bar0 + 64, st);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(g.ctas);
  cfg.blockDim = dim3(kBlockThreads);
  cfg.dynamicSmemBytes = g.smem;
  cfg.stream = st;
  cudaLaunchAttribute at;
  at.id = cudaLaunchAttributeCooperative;
  at.val.cooperative = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  e = cudaLaunchKernelEx(&cfg, jacobi_team_kernel, d, g.count, max_sweeps, svd_stall());
  return e == cudaSuccess ? cudaEventRecord(last[dev], st) : e;
}

// fallback: the FP64 sweeps of a refined group, for the sectors the refinement left
cudaError_t launch_group(const SvdSector* d_secs, const SvdGroup& g, int max_sweeps, cudaStream_t st,
                         bool fallback = false) {
  if (g.count <= 0) return cudaSuccess;
  const SvdSector* d = d_secs + g.first;
  count_launch();
  if (g.kind == kSvdSmall || (g.kind == kSvdRefine && g.cl == 1 && !fallback)) {
    if (g.kind == kSvdRefine)
      svd_small_kernel<kFrontThreads><<<g.count, kFrontThreads, g.smem_small, st>>>(d, max_sweeps);
    else
      svd_small_kernel<kSvdThreads><<<g.count, kSvdThreads, g.smem_small, st>>>(d, max_sweeps);
    return cudaGetLastError();
  }
  const int cl = g.kind == kSvdRefine && g.cl == 1 ? 2 : g.cl;      // a one-CTA front falls back to a cluster of 2
  if (g.kind == kSvdSmem) {
    jacobi_cta_kernel<<<g.count, kSvdThreads, g.smem, st>>>(d, max_sweeps);
    return cudaGetLastError();
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(g.count * cl);
  cfg.blockDim = dim3(g.kind == kSvdCluster ? kSvdThreads : kBlockThreads);
  cfg.dynamicSmemBytes = g.kind == kSvdRefine && !fallback ? g.smem_small : g.smem;
  cfg.stream = st;
  cudaLaunchAttribute at;
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = cl;
  at.val.clusterDim.y = 1;
  at.val.clusterDim.z = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  if (g.kind == kSvdTeam) return launch_teams(d, g, max_sweeps, st);
  if (g.kind == kSvdRefine && !fallback) return cudaLaunchKernelEx(&cfg, svd_front_kernel, d, g.cl, max_sweeps, svd_stall());
  if (g.kind == kSvdRefine) return cudaLaunchKernelEx(&cfg, jacobi_cluster_block_kernel<true>, d, cl, max_sweeps, svd_stall());
  if (g.kind != kSvdCluster) return cudaLaunchKernelEx(&cfg, jacobi_cluster_block_kernel<false>, d, cl, max_sweeps, svd_stall());
  return cudaLaunchKernelEx(&cfg, jacobi_cluster_kernel, d, g.cl, max_sweeps);
}

}  // namespace

// Teams instead of clusters for the block-Jacobi sectors of a batch whose largest sectors would
// run on long after the others.  A sector's work in CTA-seconds, fitted to measured sectors from
// 1551 x 47 to 796 x 796: 13.5 K^3 + 6 m n K, 9.2 m n K when wide (units of 1e-9).  Clusters end after the
// largest work / cluster size; teams are sized so that all sectors end together, at most one CTA per
// block pair of a round.  They are formed when that is less than 2/3 of the clusters' time: teams pay for
// barriers across the chip (2 us), and with hundreds of large sectors the clusters keep every SM busy.
cudaError_t form_teams(std::vector<SvdSector>& secs, std::vector<std::pair<int, int>>& key,
                       const std::vector<int64_t>& smem) {
  std::vector<size_t> who;
  int64_t need = 0;
  double total = 0.0, longest = 0.0;
  std::vector<double> work(secs.size(), 0.0);
  for (size_t k = 0; k < secs.size(); ++k) {
    if (key[k].first != kSvdClusterBlock || secs[k].F || !secs[k].teambar) continue;
    const double m = secs[k].m, n = secs[k].n, K = std::min(m, n);
    work[k] = 13.5 * K * K * K + (secs[k].wide ? 9.2 : 6.0) * m * n * K;
    who.push_back(k);
    need = std::max(need, smem[k]);
    total += work[k];
    longest = std::max(longest, work[k] / key[k].second);
  }
  if (who.empty()) return cudaSuccess;
  int dev = 0, sms = 0, coop = 0, per_sm = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
  if (e == cudaSuccess)
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, jacobi_team_kernel, kBlockThreads, (size_t)need);
  if (e != cudaSuccess) return e;
  const int cap = std::min(kMaxTeam, sms * per_sm);
  if (!coop || (int)who.size() > cap) return cudaSuccess;
  // the fewest CTAs that end sector k by time T (or one per block pair): the pairs of a round are dealt
  // out in whole turns, so only sizes that change the number of turns count
  auto size_for = [&](size_t k, double T) {
    const int pairs = key[k].second * secs[k].groups;
    const int turns = (int)std::max(1.0, std::min((double)pairs, std::floor(T * pairs / work[k])));
    return std::min(kMaxTeam, (pairs + turns - 1) / turns);
  };
  auto ctas = [&](double T) {
    int64_t s = 0;
    for (size_t k : who) s += size_for(k, T);
    return s;
  };
  double lo = total / cap, hi = total;
  while (ctas(lo) > cap && hi > 1.02 * lo) {
    const double T = 0.5 * (lo + hi);
    if (hi < 1.04 * lo) break;
    if (ctas(T) > cap) lo = T; else hi = T;
  }
  const double T = ctas(lo) <= cap ? lo : hi;
  if (ctas(T) > cap) return cudaSuccess;
  double ends = 0.0;
  for (size_t k : who) ends = std::max(ends, work[k] / size_for(k, T));
  if (ends > 2.0 / 3.0 * longest) return cudaSuccess;
  for (size_t k : who) {
    secs[k].team_size = size_for(k, T);
    secs[k].team_cl0 = key[k].second;
    key[k] = {kSvdTeam, 1};
  }
  return cudaSuccess;
}

// The kernel and the cluster size of one sector, its block pairs (groups, staged, front_staged) and the dynamic
// shared memory of the FP64 sweeps and of the front.  Host arithmetic alone; clears F where the sector is not refined.
struct SvdShape {
  int kind, cl;
  int64_t smem, small;
};
SvdShape sector_shape(SvdSector& S, const SvdTune& tune, int big_cluster) {
  SvdShape r = {};
  if (S.mode == kSvdSmem) {
    r.kind = S.small ? kSvdSmall : kSvdSmem;
    r.cl = 1;
    r.smem = svd_smem_need(S.m, S.n);
    if (S.small) r.small = std::max(r.smem, small_layout(S.m, S.n, true).total);
    return r;
  }
  const int K = std::min(S.m, S.n), bw = std::max(2, tune.bw);
  const int cn = S.wide ? K : S.n;   // Jacobi column length
  if (S.F && small_layout(S.m, S.n, false).total <= kFrontSmemMax) {
    // a one-CTA front; should the FP64 sweeps be needed, a cluster of 2 stages all its block pairs
    const int g = std::max(1, (K + bw * 2) / (2 * bw * 2));
    if (g <= kMaxStaged && block_smem_need(S.m, cn, 2, g, g) <= kBlockSmemMax) {
      S.groups = S.staged = g;
      return SvdShape{kSvdRefine, 1, block_smem_need(S.m, cn, 2, g, g), small_layout(S.m, S.n, false).total};
    }
  }
  // blocks of about tune.bw columns (6 by default); the smallest cluster (tune.cl_min,
  // then doubling up to 8 CTAs) whose CTAs can stage all of their block pairs of a round
  // at once, so that a step offers the warp groups about K / (2 cl) * bw / 2 disjoint
  // pairs; failing that, 8 CTAs staging as many pairs as fit, with more pairs per CTA
  // when a single one does not fit.  A front's blocks serve its FP32 sweeps and the FP64 sweeps that may have to
  // follow, whose columns are longer in bytes unless n is well below K: one pair of either has to fit.
  auto need = [&](int cl, int g, int gs) {
    return S.F ? front_smem_need(S.m, cn, cl, g, gs) : block_smem_need(S.m, cn, cl, g, gs);
  };
  const int64_t room = S.F ? kPairSmemMax : kBlockSmemMax;
  auto fits = [&](int cl, int g, int gs) {
    return need(cl, g, gs) <= room && block_smem_need(S.m, cn, cl, g, 1) <= kBlockSmemMax;
  };
  auto blocks = [&](int cl) {      // of a front: at most bw columns each, its 6 warps' slots a pair of them
    return S.F ? (K + 2 * bw * cl - 1) / (2 * bw * cl) : std::max(1, (K + bw * cl) / (2 * bw * cl));
  };
  int pick_cl = 0, pick_g = 0, pick_gs = 0;
  for (int cl = std::max(2, std::min(tune.cl_min, kBigCluster)); cl <= kBigCluster && !pick_cl; cl *= 2) {
    const int g = blocks(cl);
    if (g <= kMaxStaged && fits(cl, g, g)) {
      pick_cl = cl; pick_g = g; pick_gs = g;
    }
  }
  auto in_chunks = [&](int cl) {
    int g = blocks(cl);
    while (g < 64 && !fits(cl, g, 1)) ++g;
    int gs = 1;
    while (gs < std::min(g, kMaxStaged) && fits(cl, g, gs + 1)) ++gs;
    if (fits(cl, g, gs)) {
      pick_cl = cl; pick_g = g; pick_gs = gs;
    }
  };
  if (!pick_cl) in_chunks(kBigCluster);
  if (K >= tune.c16_min_k && big_cluster >= 16) in_chunks(16);
  if (K >= tune.rr_min_k || !pick_cl) {
    S.F = nullptr;        // the round-robin kernel runs in FP64 alone
    return SvdShape{kSvdCluster, big_cluster, 0, 0};
  }
  r.kind = S.F ? kSvdRefine : kSvdClusterBlock;
  r.cl = pick_cl;
  S.groups = pick_g;
  if (S.F) {
    S.front_staged = pick_gs;
    r.small = std::max<int64_t>(need(pick_cl, pick_g, pick_gs),
                                16LL * std::max(S.m, S.n));      // the QR's copy of a reflector
    while (block_smem_need(S.m, cn, pick_cl, pick_g, pick_gs) > kBlockSmemMax) --pick_gs;      // 1 fits
  }
  S.staged = pick_gs;
  r.smem = block_smem_need(S.m, cn, pick_cl, pick_g, pick_gs);
  return r;
}

cudaError_t svd_group(std::vector<SvdSector>& secs, std::vector<SvdGroup>& groups, const SvdTune& tune, bool team) {
  int big_cluster = 0;
  cudaError_t e = set_attrs(&big_cluster);
  if (e != cudaSuccess) return e;
  // every sector gets a kernel and a cluster size
  std::vector<std::pair<int, int>> key(secs.size());
  std::vector<int64_t> smem(secs.size(), 0), small(secs.size(), 0);
  for (size_t k = 0; k < secs.size(); ++k) {
    const SvdShape r = sector_shape(secs[k], tune, big_cluster);
    key[k] = {r.kind, r.cl};
    smem[k] = r.smem;
    small[k] = r.small;
  }
  if (team && (e = form_teams(secs, key, smem)) != cudaSuccess) return e;
  // group by (kind, cluster size); the most expensive sectors first inside a group
  std::vector<size_t> idx(secs.size());
  for (size_t k = 0; k < idx.size(); ++k) idx[k] = k;
  auto cost = [&](size_t k) {
    const double C = std::min(secs[k].m, secs[k].n);
    return (double)secs[k].n * C * C + (double)secs[k].m * secs[k].n * C;
  };
  std::stable_sort(idx.begin(), idx.end(), [&](size_t a, size_t b) {
    if (key[a] != key[b]) return key[a] > key[b];
    return cost(a) > cost(b);
  });
  std::vector<SvdSector> out;
  out.reserve(secs.size());
  groups.clear();
  for (size_t t = 0; t < idx.size(); ++t) {
    const size_t k = idx[t];
    if (groups.empty() || groups.back().kind != key[k].first || groups.back().cl != key[k].second) {
      SvdGroup g = {};
      g.kind = key[k].first;
      g.cl = key[k].second;
      g.smem = 0;
      g.first = (int)out.size();
      g.count = 0;
      g.max_k = g.max_n = 0;
      groups.push_back(g);
    }
    groups.back().count++;
    groups.back().smem = std::max<int>(groups.back().smem, (int)smem[k]);
    groups.back().smem_small = std::max<int>(groups.back().smem_small, (int)small[k]);
    groups.back().max_k = std::max(groups.back().max_k, std::min(secs[k].m, secs[k].n));
    groups.back().max_n = std::max(groups.back().max_n, secs[k].n);
    if (key[k].first == kSvdTeam) {
      SvdGroup& g = groups.back();
      secs[k].team_first = g.ctas;
      g.ctas += secs[k].team_size;
      if (!g.bar0 || secs[k].teambar < g.bar0) g.bar0 = secs[k].teambar;
      if (!g.bar1 || secs[k].teambar > g.bar1) g.bar1 = secs[k].teambar;
    }
    out.push_back(secs[k]);
  }
  secs.swap(out);
  return cudaSuccess;
}

cudaError_t svd_side_streams(mps_s* h, int n) {
  for (n = std::min(n, kSvdSideStreams); h->n_side < n; ++h->n_side) {
    cudaStream_t& s = h->side[h->n_side];
    cudaEvent_t& j = h->join[h->n_side];
    cudaError_t e = s ? cudaSuccess : cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking);
    if (e == cudaSuccess && !j) e = cudaEventCreateWithFlags(&j, cudaEventDisableTiming);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t launch_svd_groups(const SvdSector* d_secs, const std::vector<SvdGroup>& groups, cudaStream_t st,
                              const cudaStream_t* side, int n_side, cudaEvent_t fork, const cudaEvent_t* join,
                              int max_sweeps) {
  max_sweeps = std::max(1, std::min(max_sweeps, kJacobiMaxSweeps));   // the flag arrays hold 40 sweeps
  // group 0 on st, the others on side streams when given, all joined back into st
  cudaError_t e = cudaSuccess;
  const int ng = (int)groups.size();
  if (ng == 0) return cudaSuccess;
  const bool fan = side && n_side >= ng - 1 && ng > 1;
  // Clusters of 8 need free places on several SMs at once, so with them the one-CTA kernels, which take up to a
  // whole SM and end first, go behind the last smaller clusters instead of beside them (a layer of 77 sectors at
  // chi = 333: fronts done after 17.7 instead of 20 ms).
  auto one_cta = [&](int g) {
    return groups[g].kind <= kSvdSmall || (groups[g].kind == kSvdRefine && groups[g].cl == 1);
  };
  const bool behind = groups[0].kind == kSvdRefine && groups[0].cl == kBigCluster;
  auto lane = [&](int g) {
    while (behind && g > 1 && one_cta(g)) --g;
    return g;
  };
  if (fan) {      // only the streams that get work: each is joined below, as a capture wants
    if ((e = cudaEventRecord(fork, st)) != cudaSuccess) return e;
    for (int g = 1; g < ng; ++g)
      if (lane(g) == g && (e = cudaStreamWaitEvent(side[g - 1], fork, 0)) != cudaSuccess) return e;
  }
  for (int g = 0; g < ng; ++g) {
    cudaStream_t s = (fan && g > 0) ? side[lane(g) - 1] : st;
    if ((e = launch_group(d_secs, groups[g], max_sweeps, s)) != cudaSuccess) return e;
  }
  auto joined = [&](int g, cudaStream_t into) -> cudaError_t {
    cudaStream_t from = side[lane(g) - 1];
    if (from == into) return cudaSuccess;
    cudaError_t e2 = cudaEventRecord(join[g - 1], from);
    return e2 == cudaSuccess ? cudaStreamWaitEvent(into, join[g - 1], 0) : e2;
  };
  auto refine = [&](int g0, int g1, cudaStream_t s) -> cudaError_t {      // groups g0 .. g1 - 1, their fronts done
    int count = 0, max_k = 0, max_n = 0;
    for (int g = g0; g < g1; ++g) {
      count += groups[g].count;
      max_k = std::max(max_k, groups[g].max_k);
      max_n = std::max(max_n, groups[g].max_n);
    }
    cudaError_t e2 = launch_refine(d_secs + groups[g0].first, count, max_k, max_n, s);
    for (int g = g0; g < g1 && e2 == cudaSuccess; ++g) e2 = launch_group(d_secs, groups[g], max_sweeps, s, true);
    return e2;
  };
  // The refined groups come first.  Clusters of 8 run on when the other fronts are done, and leave SMs free by then,
  // so those sectors are refined meanwhile; without clusters of 8 all are refined together.
  int nr = 0;
  while (nr < ng && groups[nr].kind == kSvdRefine) ++nr;
  const int first = fan && behind && nr > 1 ? 1 : 0;      // the first group of the refinement beside
  if (first) {
    cudaStream_t s = side[lane(nr - 1) - 1];
    for (int g = 1; g < nr; ++g)
      if ((e = joined(g, s)) != cudaSuccess) return e;
    if ((e = refine(1, nr, s)) != cudaSuccess || (e = refine(0, 1, st)) != cudaSuccess) return e;
  } else {
    if (fan)
      for (int g = 1; g < nr; ++g)
        if ((e = joined(g, st)) != cudaSuccess) return e;
    if (nr > 0 && (e = refine(0, nr, st)) != cudaSuccess) return e;
  }
  if (fan)
    for (int g = first ? 1 : std::max(nr, 1); g < ng; ++g)
      if ((e = joined(g, st)) != cudaSuccess) return e;
  return cudaSuccess;
}

bool svd_layout(int ns, const int* m, const int* n, SvdScratchLayout& L, int cluster_min_k, const char* exact,
                bool team) {
  if (cluster_min_k < 0) cluster_min_k = svd_cluster_min_k();
  L.mode.assign(ns, kSvdSmem);
  L.work_off.assign(ns, -1);
  L.v_off.assign(ns, -1);
  L.norm_off.assign(ns, -1);
  L.ord_off.assign(ns, -1);
  L.flag_off.assign(ns, -1);
  L.piv_off.assign(ns, -1);
  L.wide.assign(ns, 0);
  L.exact.assign(ns, 0);
  L.small.assign(ns, 0);
  L.bar_off = -1;
  const int members = team ? kMaxTeam : kMaxCluster;
  L.w2_off.assign(ns, -1);
  L.yt_off.assign(ns, -1);
  for (auto* v : {&L.f32_off, &L.n32_off, &L.vd_off, &L.gm_off, &L.a1_off, &L.sel_off, &L.j_off, &L.v_off2, &L.misc_off})
    v->assign(ns, -1);
  L.smem = 0;
  // FP64 updates refine at every size unless the caller has asked for FP64 sweeps, at all sizes (0) or up to a size
  // above the default
  const int set_k = svd_mixed_min_k();
  const bool any_k = set_k > 0 && set_k <= kMixedMinK;
  const int own_k = any_k ? kRefineMinK : set_k;
  int64_t off = 0;
  auto a256 = [](int64_t x) { return (x + 255) & ~int64_t(255); };
  for (int k = 0; k < ns; ++k) {
    if (m[k] < 1 || n[k] < 1) return false;
    const int64_t need = svd_smem_need(m[k], n[k]);
    L.exact[k] = exact && exact[k];
    // a front's CTAs hold a copy of the QR's reflector; longer columns keep the FP32 start of the other sectors
    const bool refine = !L.exact[k] && own_k > 0 && std::min(m[k], n[k]) >= own_k &&
                        16LL * std::max(m[k], n[k]) <= kBlockSmemMax;
    if (need <= kSvdSmemMax && std::min(m[k], n[k]) < cluster_min_k && !refine) {
      L.small[k] = !L.exact[k] && any_k && std::min(m[k], n[k]) <= kSmallK &&
                   small_layout(m[k], n[k], true).total <= kSvdSmemMax;
      L.smem = std::max<int>(L.smem, (int)need);
      continue;
    }
    const int64_t M = m[k], N = n[k], Kk = std::min(m[k], n[k]);
    L.mode[k] = kSvdCluster;
    L.work_off[k] = off; off = a256(off + 16 * M * odd_ld(n[k]));
    L.v_off[k] = off;    off = a256(off + 16 * M);                      // Householder vector
    L.norm_off[k] = off; off = a256(off + 8 * (2 * N + Kk));            // nu, nu0, nrm
    L.ord_off[k] = off;  off = a256(off + 4 * (N + Kk));                // perm, ord
    L.flag_off[k] = off; off = a256(off + 4 * (kJacobiMaxSweeps + 1 + members));       // flags, pivot index
    L.piv_off[k] = off;  off = a256(off + 8 * (members + 2));           // pivot value, scalars
    const bool wide = 4LL * n[k] >= 5LL * m[k];   // the Jacobi sweeps run on the K x K factor R2
    L.wide[k] = wide;
    if (refine) {   // FP32 start and refinement (svd_front, k_refine.cu); the FP64 sweeps that may
                    // follow use the same space (svd_fill_scratch)
      const int64_t jlen = wide ? Kk : N;
      L.j_off[k] = off;    off = a256(off + 16 * N * Kk);
      L.a1_off[k] = off;   off = a256(off + 16 * odd_ld(n[k]) * Kk);
      L.v_off2[k] = off;   off = a256(off + 2 * 16 * Kk * odd_ld((int)Kk));
      L.misc_off[k] = off; off = a256(off + 64 + 16 + 8 * Kk + 4 * (4 * Kk + 1) + 16);
      off = a256(off + 8 * (jlen + Kk + 2) * Kk);      // F, behind the small arrays
      L.w2_off[k] = L.v_off2[k] + 16 * Kk * odd_ld((int)Kk);
      L.yt_off[k] = L.a1_off[k];
    } else {
      if (wide) {
        L.w2_off[k] = off; off = a256(off + 16 * Kk * odd_ld((int)Kk));     // R2 / Jacobi matrix
        L.yt_off[k] = off; off = a256(off + 16 * N * Kk);                   // Q2 applied to its columns
      }
      if (set_k > 0 && Kk >= set_k) {   // FP32 sweeps first (see mixed_precondition)
        const int64_t jlen = wide ? Kk : N, jld = wide ? odd_ld((int)Kk) : odd_ld(n[k]);
        L.f32_off[k] = off; off = a256(off + 8 * (jlen + Kk + 2) * Kk);
        L.n32_off[k] = off; off = a256(off + 4 * Kk);
        L.vd_off[k] = off;  off = a256(off + 16 * Kk * Kk);
        L.gm_off[k] = off;  off = a256(off + 16 * Kk * Kk);
        L.a1_off[k] = off;  off = a256(off + 16 * jld * Kk);
        L.sel_off[k] = off; off = a256(off + 4 * (Kk + 1));
      }
    }
  }
  if (team) {   // one 64-byte line a sector for the barrier of its team
    L.bar_off = off;
    off = a256(off + 64LL * ns);
  }
  L.total = off;
  return true;
}

void svd_fill_scratch(SvdSector& S, const SvdScratchLayout& L, int k, char* base) {
  S.mode = L.mode[k];
  S.small = L.small[k];
  S.F = nullptr;
  S.fp32_sweeps = svd_mixed_sweeps();
  if (S.mode != kSvdCluster) return;
  S.work = reinterpret_cast<double2*>(base + L.work_off[k]);
  S.uwork = reinterpret_cast<double2*>(base + L.v_off[k]);
  S.norms = reinterpret_cast<double*>(base + L.norm_off[k]);
  S.order = reinterpret_cast<int*>(base + L.ord_off[k]);
  S.flags = reinterpret_cast<int*>(base + L.flag_off[k]);
  S.pivv = reinterpret_cast<double*>(base + L.piv_off[k]);
  S.wide = L.wide[k];
  if (S.wide) {
    S.work2 = reinterpret_cast<double2*>(base + L.w2_off[k]);
    S.ytmp = reinterpret_cast<double2*>(base + L.yt_off[k]);
  }
  S.f32 = nullptr;
  S.fp32_sweeps = svd_mixed_sweeps();
  S.F = nullptr;
  S.teambar = L.bar_off >= 0 ? reinterpret_cast<unsigned*>(base + L.bar_off + 64LL * k) : nullptr;
  if (L.f32_off[k] >= 0) {
    S.f32 = reinterpret_cast<float2*>(base + L.f32_off[k]);
    S.nrm32 = reinterpret_cast<float*>(base + L.n32_off[k]);
    S.vd = reinterpret_cast<double2*>(base + L.vd_off[k]);
    S.gm = reinterpret_cast<double2*>(base + L.gm_off[k]);
    S.a1 = reinterpret_cast<double2*>(base + L.a1_off[k]);
    S.sel = reinterpret_cast<int*>(base + L.sel_off[k]);
  }
  if (L.misc_off[k] >= 0) {
    const int64_t K = std::min(S.m, S.n);
    S.J = reinterpret_cast<double2*>(base + L.j_off[k]);
    S.A0 = S.work;
    S.A1 = reinterpret_cast<double2*>(base + L.a1_off[k]);
    S.V0 = reinterpret_cast<double2*>(base + L.v_off2[k]);
    S.V1 = S.V0 + K * odd_ld((int)K);
    char* p = base + L.misc_off[k];
    S.rstate = reinterpret_cast<int*>(p);          p += 64;
    S.rfloor2 = reinterpret_cast<double*>(p);      p += 16;
    S.rnorm = reinterpret_cast<double*>(p);        p += 8 * K;
    S.cexp = reinterpret_cast<int*>(p);            p += 4 * K;
    S.vexp = reinterpret_cast<int*>(p);            p += 4 * K;
    S.nrm32 = reinterpret_cast<float*>(p);         p += 4 * K;
    S.sel = reinterpret_cast<int*>(p);             p += 4 * (K + 1);
    S.F = reinterpret_cast<float2*>(base + ((p - base + 255) & ~int64_t(255)));
    // for the FP64 sweeps that go on from J and V32 (copied to work and vd first): J's space holds the Gram matrix; J V is in
    // A1's, or in F's where a wide sector has Q2's product in A1's (R2 is in V1's)
    S.vd = S.V0;
    S.gm = S.J;
    S.a1 = S.wide ? reinterpret_cast<double2*>(S.F) : S.A1;
  }
}

namespace {
std::atomic<int> g_mixed_min_k{kMixedMinK};
std::atomic<int> g_mixed_sweeps{8};
std::atomic<int> g_cluster_min_k{1 << 30};
std::atomic<int> g_svd_stall{0};
}
int svd_stall() { return g_svd_stall.load(); }
int svd_mixed_min_k() { return g_mixed_min_k.load(); }
int svd_cluster_min_k() { return g_cluster_min_k.load(); }
int svd_mixed_sweeps() { return g_mixed_sweeps.load(); }

}  // namespace mps

extern "C" int mps_svd_mixed_min_k(int min_k) {
  if (min_k < 0) return MPS_EINVAL;
  mps::g_mixed_min_k.store(min_k);
  return MPS_OK;
}

extern "C" int mps_svd_inject_stall(int what) {
  if (what & ~(mps::kStallBlocks | mps::kStallFronts)) return MPS_EINVAL;
  mps::g_svd_stall.store(what);
  return MPS_OK;
}

extern "C" int mps_svd_cluster_min_k(int min_k) {
  if (min_k != 0 && min_k < 16) return MPS_EINVAL;
  mps::g_cluster_min_k.store(min_k == 0 ? (1 << 30) : min_k);
  return MPS_OK;
}

extern "C" int mps_svd_mixed_sweeps(int max_sweeps) {
  if (max_sweeps < 1 || max_sweeps > mps::kJacobiMaxSweeps) return MPS_EINVAL;
  mps::g_mixed_sweeps.store(max_sweeps);
  return MPS_OK;
}

using namespace mps;

extern "C" int64_t mps_svd_path_work_bytes(int n_sectors, const int* m, const int* n, int keep_phases) {
  if (n_sectors < 0 || (n_sectors > 0 && (!m || !n))) return -1;
  SvdScratchLayout L;
  const std::vector<char> exact(n_sectors, keep_phases != 0);
  if (!svd_layout(n_sectors, m, n, L, -1, exact.data())) return -1;
  return ((int64_t)sizeof(SvdSector) * n_sectors + 255) / 256 * 256 + L.total;
}

extern "C" int64_t mps_svd_work_bytes(int n_sectors, const int* m, const int* n) {
  return mps_svd_path_work_bytes(n_sectors, m, n, 0);
}

extern "C" int mps_svd_sector_plan(int m, int n, int keep_phases, int* path, int* ctas, int* block_pairs,
                                   int* staged) {
  SvdScratchLayout L;
  const char exact = keep_phases != 0;
  if (m < 1 || n < 1 || !svd_layout(1, &m, &n, L, -1, &exact)) return MPS_EINVAL;
  alignas(256) static char none[256];      // addresses are formed from it, nothing is read or written
  SvdSector S = {};
  S.m = m;
  S.n = n;
  svd_fill_scratch(S, L, 0, none);
  SvdTune tune;
  svd_forced_tune(tune);
  const SvdShape r = sector_shape(S, tune, kMaxCluster);
  const bool start = r.kind == kSvdClusterBlock && S.f32 && std::min(m, n) >= 2;
  if (path)
    *path = r.kind == kSvdRefine || r.kind == kSvdSmall
                ? MPS_SVD_REFINED
                : MPS_SVD_SWEEPS | (start ? MPS_SVD_FP32_START : 0) | (r.kind == kSvdCluster ? MPS_SVD_ROUND_ROBIN : 0);
  if (ctas) *ctas = r.cl;
  if (block_pairs) *block_pairs = S.groups;
  if (staged) *staged = S.front_staged ? S.front_staged : S.staged;
  return MPS_OK;
}

namespace {
// The sectors of one call, in scratch laid out by L behind desc bytes of descriptors.
struct SectorCall {
  int n_sectors;
  const int *m, *n;
  const double* d_mats;
  const int64_t* mat_off;
  const double* d_rowscale;
  const int64_t* row_off;
  double* d_sigma;
  const int64_t* sig_off;
  double* d_y;
  const int64_t* y_off;
  int *d_status, *d_path;
  bool valid() const {
    return n_sectors > 0 && m && n && d_mats && mat_off && d_sigma && sig_off && d_y && y_off && d_status &&
           !(d_rowscale && !row_off);
  }
  int64_t desc() const { return ((int64_t)sizeof(SvdSector) * n_sectors + 255) / 256 * 256; }
  int run(const SvdScratchLayout& L, void* d_work, cudaStream_t st) const {
    std::vector<SvdSector> cta, cl;
    char* base = (char*)d_work + desc();
    for (int k = 0; k < n_sectors; ++k) {
      SvdSector S = {};
      S.theta = reinterpret_cast<const double2*>(d_mats) + mat_off[k];
      S.rowscale = d_rowscale ? d_rowscale + row_off[k] : nullptr;
      S.m = m[k];
      S.n = n[k];
      svd_fill_scratch(S, L, k, base);
      S.sigma = d_sigma + sig_off[k];
      S.Y = reinterpret_cast<double2*>(d_y) + y_off[k];
      S.status = d_status + k;
      S.path = d_path ? d_path + k : nullptr;
      (S.mode == kSvdCluster ? cl : cta).push_back(S);
    }
    std::vector<SvdSector> all(cta);
    all.insert(all.end(), cl.begin(), cl.end());
    std::vector<SvdGroup> groups;
    SvdTune tune;
    svd_forced_tune(tune);
    if (svd_group(all, groups, tune) != cudaSuccess) return MPS_ECUDA;
    if (cudaMemcpyAsync(d_work, all.data(), sizeof(SvdSector) * all.size(), cudaMemcpyHostToDevice, st) !=
        cudaSuccess)
      return MPS_ECUDA;
    const SvdSector* d_all = reinterpret_cast<const SvdSector*>(d_work);
    if (launch_svd_groups(d_all, groups, st, nullptr, 0, nullptr, nullptr) != cudaSuccess) return MPS_ECUDA;
    // the descriptors came from pageable host memory: finish before returning
    return cudaStreamSynchronize(st) == cudaSuccess ? MPS_OK : MPS_ECUDA;
  }
};
}  // namespace

extern "C" int mps_svd_sectors_path(int n_sectors, const int* m, const int* n,
                                    const double* d_mats, const int64_t* mat_off,
                                    const double* d_rowscale, const int64_t* row_off,
                                    double* d_sigma, const int64_t* sig_off,
                                    double* d_y, const int64_t* y_off,
                                    int* d_status, int keep_phases, int* d_path,
                                    void* d_work, int64_t work_bytes, void* cuda_stream) {
  if (n_sectors == 0) return MPS_OK;
  const SectorCall C{n_sectors, m,       n,   d_mats, mat_off,  d_rowscale, row_off,
                     d_sigma,   sig_off, d_y, y_off,  d_status, d_path};
  if (!C.valid() || !d_work) return MPS_EINVAL;
  SvdScratchLayout L;
  const std::vector<char> exact(n_sectors, keep_phases != 0);
  if (!svd_layout(n_sectors, m, n, L, -1, exact.data())) return MPS_EINVAL;
  if (work_bytes < C.desc() + L.total) return MPS_EINVAL;
  return C.run(L, d_work, (cudaStream_t)cuda_stream);
}

extern "C" int mps_svd_sectors(int n_sectors, const int* m, const int* n,
                               const double* d_mats, const int64_t* mat_off,
                               const double* d_rowscale, const int64_t* row_off,
                               double* d_sigma, const int64_t* sig_off,
                               double* d_y, const int64_t* y_off,
                               int* d_status, void* d_work, int64_t work_bytes, void* cuda_stream) {
  return mps_svd_sectors_path(n_sectors, m, n, d_mats, mat_off, d_rowscale, row_off, d_sigma, sig_off, d_y, y_off,
                              d_status, 0, nullptr, d_work, work_bytes, cuda_stream);
}

// ---------------------------------------------------------------------------
// Allocation-free variant: the scratch is a file-scope device array.  In host
// code the array's name is only a host-side stand-in, so its device address is
// looked up once per device (with that device current) and passed to the
// kernels; device code never names it.
// ---------------------------------------------------------------------------
namespace {
static __device__ __align__(256) unsigned char g_noalloc_scratch[MPS_NOALLOC_SCRATCH_BYTES];
constexpr int kNoAllocMaxDevices = 64;
std::mutex g_noalloc_mutex;
void* g_noalloc_addr[kNoAllocMaxDevices] = {};
}  // namespace

extern "C" int mps_svd_sectors_noalloc(int n_sectors, const int* m, const int* n,
                                       const double* d_mats, const int64_t* mat_off,
                                       const double* d_rowscale, const int64_t* row_off,
                                       double* d_sigma, const int64_t* sig_off,
                                       double* d_y, const int64_t* y_off,
                                       int* d_status, void* cuda_stream) {
  if (n_sectors == 0) return MPS_OK;
  const SectorCall C{n_sectors, m,       n,   d_mats, mat_off,  d_rowscale, row_off,
                     d_sigma,   sig_off, d_y, y_off,  d_status, nullptr};
  if (!C.valid()) return MPS_EINVAL;
  SvdScratchLayout L;
  if (!svd_layout(n_sectors, m, n, L)) return MPS_EINVAL;
  if (C.desc() + L.total > (int64_t)MPS_NOALLOC_SCRATCH_BYTES) {   // the FP64 sweeps need less scratch
    const std::vector<char> plain(n_sectors, 1);
    if (!svd_layout(n_sectors, m, n, L, -1, plain.data())) return MPS_EINVAL;
  }
  if (C.desc() + L.total > (int64_t)MPS_NOALLOC_SCRATCH_BYTES) return MPS_ENOMEM;   // over the fixed scratch
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess) return MPS_ECUDA;
  if (dev < 0 || dev >= kNoAllocMaxDevices) return MPS_EINVAL;
  void* d_work = nullptr;
  {
    std::lock_guard<std::mutex> lock(g_noalloc_mutex);
    if (!g_noalloc_addr[dev]) {
      void* p = nullptr;
      if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess || !p) return MPS_ECUDA;
      g_noalloc_addr[dev] = p;
    }
    d_work = g_noalloc_addr[dev];
  }
  return C.run(L, d_work, (cudaStream_t)cuda_stream);
}
