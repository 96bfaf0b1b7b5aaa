// Sector GEMMs of the two-site update, FP64 complex on the CUDA cores.
//
// K1 (theta_kernel): for every (l, r) pair of one update,
//     Theta'(c)[l, r] += G_n[l - c, l - m] * (B^[s][l, m] . B^[s+1][m, r])
// summed over the middle charges m, for every new middle charge c of the pair
// (n = l - r).  This is the block-sparse construction of Theta of Sec. II: each
// product B[l,m] B[m,r] is formed once and mixed into all output charges c
// in registers, so the GEMM work is that of the (l, m, r) triples alone.
//
// K4 (gemm_kernel, scatter_kernel, lambda_kernel): reassembly after truncation,
//     B^[s][l, c]   = Theta'(c)[rows of l] . Y(c)[:, kept] / |S_kept|
//     B^[s+1][c, r] = Y(c)[cols of r, kept]^dag
//     lambda^[s+1]  = S_kept / |S_kept|
// Sites are written in charge-sorted block order with coalesced row-major stores.
//
// GB300 note: FP64 runs at 1.2 TFLOP/s on this part (2 FMA per clock and SM, measured), so these kernels
// are bound by the FP64 pipe, and a block's time is its FMAs on the SMs that share it.  A CTA of 64
// threads computes 8 x 8 outputs, one a thread: blocks of 10-100 states spread over many SMs and
// ragged edges cost least padding.  The operands a tile re-reads come from L2 (4 bytes a complex FMA).
// Stages of 16 k are copied asynchronously, the next one (of the next middle charge, too) while the present
// one is used.  64 x 64 tiles of 256 threads took 73 us (Theta) and 67 us (reassembly) on a chi = 64 XXZ
// layer of 35-state blocks, and ran at 510-570 GFLOP/s on a chi = 512 Bose-Hubbard layer (7.7 and 6.6 ms);
// these take 15 and 9 us, and 3.9 and 3.4 ms (1.0-1.1 TFLOP/s, 80-87% of the FP64 peak).
#include <algorithm>

#include "mps_internal.h"

namespace mps {
namespace {

constexpr int kS = 8;              // rows and columns of a CTA's outputs
constexpr int kK = 16;             // K chunk staged in shared memory
constexpr int kThreads = kS * kS;

struct TileSmem {
  double2 A[2][kS][kK + 1];        // +1: the rows that a warp reads together do not share banks
  double2 B[2][kK][kS];
};

__device__ __forceinline__ void cfma(double2& acc, double2 a, double2 b) {
  acc.x = fma(a.x, b.x, acc.x);
  acc.x = fma(-a.y, b.y, acc.x);
  acc.y = fma(a.x, b.y, acc.y);
  acc.y = fma(a.y, b.x, acc.y);
}

// 16-byte copy into shared memory, zeros when ok is false
__device__ __forceinline__ void copy16(double2* dst, const double2* src, bool ok) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 16, %2;\n" ::"r"((uint32_t)__cvta_generic_to_shared(dst)),
               "l"(src), "r"(ok ? 16 : 0)
               : "memory");
}

// One product of a tile: A (M x K) and B (K x N) with general strides.
struct Product {
  const double2 *A, *B;
  int sar, sac, sbr, sbc, M, N, K;
};

__device__ __forceinline__ void stage(const Product& P, int row0, int col0, int k0, int buf, TileSmem& sm) {
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int e = threadIdx.x + h * kThreads;
    const int ar = P.sac == 1 ? e >> 4 : e & 7, ak = P.sac == 1 ? e & 15 : e >> 3;
    const bool oka = row0 + ar < P.M && k0 + ak < P.K;
    copy16(&sm.A[buf][ar][ak], oka ? P.A + (int64_t)(row0 + ar) * P.sar + (int64_t)(k0 + ak) * P.sac : P.A, oka);
    const int bk = P.sbc == 1 ? e >> 3 : e & 15, bc = P.sbc == 1 ? e & 7 : e >> 4;
    const bool okb = col0 + bc < P.N && k0 + bk < P.K;
    copy16(&sm.B[buf][bk][bc], okb ? P.B + (int64_t)(k0 + bk) * P.sbr + (int64_t)(col0 + bc) * P.sbc : P.B, okb);
  }
  asm volatile("cp.async.commit_group;\n" ::: "memory");
}

// The thread's output of product P, whose first stage is on its way into buffer buf; the first stage of Q
// follows when more is set.  on: the thread's warp has rows inside the block.
__device__ __forceinline__ double2 product(const Product& P, const Product& Q, bool more, int row0, int col0, int& buf,
                                           bool on, TileSmem& sm) {
  const int tx = threadIdx.x & 7, ty = threadIdx.x >> 3;
  double p0 = 0.0, q0 = 0.0, r0 = 0.0, s0 = 0.0, p1 = 0.0, q1 = 0.0, r1 = 0.0, s1 = 0.0;
  for (int k0 = 0; k0 < P.K; k0 += kK) {
    const int kc = min(kK, P.K - k0);
    bool next = true;
    if (k0 + kK < P.K) stage(P, row0, col0, k0 + kK, buf ^ 1, sm);
    else if (more) stage(Q, row0, col0, 0, buf ^ 1, sm);
    else next = false;
    if (next) asm volatile("cp.async.wait_group 1;\n" ::: "memory");
    else asm volatile("cp.async.wait_group 0;\n" ::: "memory");
    __syncthreads();
    if (on) {
      int kk = 0;
#pragma unroll 4
      for (; kk + 1 < kc; kk += 2) {      // eight chains over the pipe's 64-cycle latency
        const double2 a = sm.A[buf][ty][kk], b = sm.B[buf][kk][tx];
        const double2 a1 = sm.A[buf][ty][kk + 1], b1 = sm.B[buf][kk + 1][tx];
        p0 = fma(a.x, b.x, p0);
        q0 = fma(a.y, b.y, q0);
        r0 = fma(a.x, b.y, r0);
        s0 = fma(a.y, b.x, s0);
        p1 = fma(a1.x, b1.x, p1);
        q1 = fma(a1.y, b1.y, q1);
        r1 = fma(a1.x, b1.y, r1);
        s1 = fma(a1.y, b1.x, s1);
      }
      if (kk < kc) {
        const double2 a = sm.A[buf][ty][kk], b = sm.B[buf][kk][tx];
        p0 = fma(a.x, b.x, p0);
        q0 = fma(a.y, b.y, q0);
        r0 = fma(a.x, b.y, r0);
        s0 = fma(a.y, b.x, s0);
      }
    }
    __syncthreads();
    buf ^= 1;
  }
  return make_double2((p0 + p1) - (q0 + q1), (r0 + r1) + (s0 + s1));
}

// blockIdx.x: a tile of kTile x kTile outputs of the task list, blockIdx.y: the kS x kS part of it
// (sub parts a row).
__global__ void __launch_bounds__(kThreads) theta_kernel(const ThetaTask* __restrict__ tasks,
                                                         const TileRef* __restrict__ tiles, int sub) {
  __shared__ TileSmem sm;
  const TileRef tr = tiles[blockIdx.x];
  const ThetaTask& T = tasks[tr.task];
  const int row0 = tr.ti * kTile + (blockIdx.y / sub) * kS, col0 = tr.tj * kTile + (blockIdx.y % sub) * kS;
  const int Dl = T.Dl, Dr = T.Dr, nc = T.nc, sn = T.sn, nm = T.nm;
  if (row0 >= Dl || col0 >= Dr) return;
  const int r = row0 + (threadIdx.x >> 3), c = col0 + (threadIdx.x & 7);
  const bool on = row0 + ((threadIdx.x >> 3) & ~3) < Dl;
  auto at = [&](int mi) { return Product{T.A[mi], T.B[mi], T.Dm[mi], 1, Dr, 1, Dl, Dr, T.Dm[mi]}; };
  double2 out[MPS_MAX_D];
#pragma unroll
  for (int k = 0; k < MPS_MAX_D; ++k) out[k] = make_double2(0.0, 0.0);
  int buf = 0;
  Product P = at(0);
  stage(P, row0, col0, 0, 0, sm);
  for (int mi = 0; mi < nm; ++mi) {
    const bool more = mi + 1 < nm;
    const Product Q = at(more ? mi + 1 : mi);
    const double2 v = product(P, Q, more, row0, col0, buf, on, sm);
    // mix this product into every output charge of the (l, r) pair
    if (on) {
#pragma unroll
      for (int k = 0; k < MPS_MAX_D; ++k)
        if (k < nc) cfma(out[k], T.gate[T.go[k] * sn + T.gi[mi]], v);
    }
    P = Q;
  }
  if (r < Dl && c < Dr) {
#pragma unroll
    for (int k = 0; k < MPS_MAX_D; ++k)
      if (k < nc) T.out[k][(int64_t)r * T.ldo[k] + c] = out[k];
  }
}

__global__ void __launch_bounds__(kThreads) gemm_kernel(const GemmTask* __restrict__ tasks,
                                                        const TileRef* __restrict__ tiles, int sub) {
  __shared__ TileSmem sm;
  const TileRef tr = tiles[blockIdx.x];
  const GemmTask& T = tasks[tr.task];
  const int row0 = tr.ti * kTile + (blockIdx.y / sub) * kS, col0 = tr.tj * kTile + (blockIdx.y % sub) * kS;
  if (row0 >= T.M || col0 >= T.N) return;
  const int r = row0 + (threadIdx.x >> 3), c = col0 + (threadIdx.x & 7);
  const Product P{T.A, T.B, T.sar, T.sac, T.sbr, T.sbc, T.M, T.N, T.K};
  int buf = 0;
  stage(P, row0, col0, 0, 0, sm);
  const double2 v = product(P, P, false, row0, col0, buf, row0 + ((threadIdx.x >> 3) & ~3) < T.M, sm);
  if (r < T.M && c < T.N) T.C[(int64_t)r * T.ldc + c] = make_double2(T.alpha * v.x, T.alpha * v.y);
}

// One flat element per thread; tasks are sorted by their first element index.
__global__ void scatter_kernel(const ScatterTask* __restrict__ tasks, int n_tasks, int64_t n_elems) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n_elems;
       e += (int64_t)gridDim.x * blockDim.x) {
    int lo = 0, hi = n_tasks - 1;
    while (lo < hi) {                       // last task with first <= e
      int mid = (lo + hi + 1) >> 1;
      if (tasks[mid].first <= e) lo = mid; else hi = mid - 1;
    }
    const ScatterTask& T = tasks[lo];
    const int64_t idx = e - T.first;
    const int j = (int)(idx / T.Dr), b = (int)(idx % T.Dr);
    const double2 y = T.Y[(int64_t)(T.coff + b) + (int64_t)j * T.n];
    T.out[idx] = make_double2(y.x, -y.y);
  }
}

__global__ void lambda_kernel(const LambdaTask* __restrict__ tasks) {
  const LambdaTask& T = tasks[blockIdx.x];
  for (int j = threadIdx.x; j < T.k; j += blockDim.x) T.lambda[j] = T.sigma[j] * T.scale;
}

}  // namespace

// parts of kS along an edge of the largest tile
inline int parts(int n) { return (std::min(n, kTile) + kS - 1) / kS; }

cudaError_t launch_theta(const ThetaTask* d_tasks, const TileRef* d_tiles, int n_tiles, int max_rows, int max_cols,
                         cudaStream_t st) {
  if (n_tiles <= 0) return cudaSuccess;
  count_launch();
  theta_kernel<<<dim3(n_tiles, parts(max_rows) * parts(max_cols)), kThreads, 0, st>>>(d_tasks, d_tiles,
                                                                                      parts(max_cols));
  return cudaGetLastError();
}

cudaError_t launch_gemm(const GemmTask* d_tasks, const TileRef* d_tiles, int n_tiles, int max_rows, int max_cols,
                        cudaStream_t st) {
  if (n_tiles <= 0) return cudaSuccess;
  count_launch();
  gemm_kernel<<<dim3(n_tiles, parts(max_rows) * parts(max_cols)), kThreads, 0, st>>>(d_tasks, d_tiles,
                                                                                     parts(max_cols));
  return cudaGetLastError();
}

cudaError_t launch_scatter(const ScatterTask* d_tasks, int n_tasks, int64_t n_elems, cudaStream_t st) {
  if (n_tasks <= 0 || n_elems <= 0) return cudaSuccess;
  int64_t blocks = (n_elems + 255) / 256;
  if (blocks > 152 * 16) blocks = 152 * 16;
  count_launch();
  scatter_kernel<<<(int)blocks, 256, 0, st>>>(d_tasks, n_tasks, n_elems);
  return cudaGetLastError();
}

cudaError_t launch_lambda(const LambdaTask* d_tasks, int n_tasks, cudaStream_t st) {
  if (n_tasks <= 0) return cudaSuccess;
  count_launch();
  lambda_kernel<<<n_tasks, 128, 0, st>>>(d_tasks);
  return cudaGetLastError();
}

}  // namespace mps
