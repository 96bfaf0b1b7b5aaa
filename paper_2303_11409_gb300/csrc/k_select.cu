// Global top-chi truncation across all charge sectors of one update (K3).
//
// Sec. II bounds every bond by chi; the truncation is global over the middle
// charges.  Rule (the paper is silent on details; the same rule is in the
// oracle): candidates are sigma > cutoff * |sigma|_2 (strict).  If at most chi
// candidates exist all are kept.  Otherwise v = the chi-th largest candidate;
// values above v + tau are kept, values within [v - tau, v + tau] are ties and
// are taken in (charge ascending, index ascending) order until chi are kept,
// tau = 1e-11 * sigma_max.  Each sector's kept set is a prefix of its
// descending list, so the result is one count per sector.
//
// One CTA per update.  The spectra are staged in shared memory (those of up to kSelSectors sectors and
// kSelValues values; larger ones are read where they are).  v is searched between the cutoff and the largest value by
// its bit pattern: a round counts the values above 2^p - 1 thresholds by binary searches, one a thread, so the range
// shrinks 2^p-fold (p = 1 to 5, by the number of sectors).  It takes a warp reduction, a few atomics and one barrier a
// round, whatever the spectra.  One update, us, by the bisection with two searches a sector and a block sum in each of
// 64 rounds | by letting every value search its own place | so: 20 sectors of 20 values 111 | 62 | 36, 30 of 150
// 172 | 211 | 47, 30 of 600 226 | 1643 | 72, 600 of 8 917 | 16657 | 476, 16 of 280 equal values 158 | 4015 | 41.
// All sums are fixed-order block reductions (deterministic).
#include "mps_internal.h"

namespace mps {
namespace {

constexpr int kSelThreads = 256;
constexpr int kSelSectors = 256, kSelValues = 4608;

// red[t] + red[t + 128], then + 64, ..., + 1: the sum of all threads' v
template <typename T>
__device__ T block_sum(T v, T* red) {
  const int tid = threadIdx.x;
  red[tid] = v;
  __syncthreads();
  for (int s = kSelThreads / 2; s >= 32; s >>= 1) {
    if (tid < s) {
      v += red[tid + s];
      red[tid] = v;
    }
    __syncthreads();
  }
  if (tid < 32) {
    for (int s = 16; s; s >>= 1) v += __shfl_down_sync(0xffffffffu, v, s);
    if (tid == 0) red[0] = v;
  }
  __syncthreads();
  const T r = red[0];
  __syncthreads();
  return r;
}

// Singular values are not negative, so their bit patterns order like the values; integer comparisons
// keep the searches off the FP64 pipe (where one costs a warp 64 cycles).
__device__ __forceinline__ long long bits(double x) { return __double_as_longlong(x); }
// number of entries of a descending array whose bits are >= b
__device__ __forceinline__ int count_from(const double* a, int k, long long b) {
  int lo = 0, hi = k;
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    if (bits(a[mid]) >= b) lo = mid + 1; else hi = mid;
  }
  return lo;
}
// number of entries of a descending array that are > x, and that are >= x
__device__ int count_gt(const double* a, int k, double x) { return x < 0.0 ? k : count_from(a, k, bits(x) + 1); }
__device__ int count_ge(const double* a, int k, double x) { return x <= 0.0 ? k : count_from(a, k, bits(x)); }

__global__ void __launch_bounds__(kSelThreads) select_kernel(const SelectSector* __restrict__ secs,
                                                             const SelectTask* __restrict__ tasks,
                                                             int* __restrict__ kept,
                                                             SelectResult* __restrict__ res) {
  __shared__ double dred[kSelThreads];
  __shared__ long long ired[kSelThreads];
  __shared__ double s_val[kSelValues];
  __shared__ const double* s_sig[kSelSectors];
  __shared__ int s_k[kSelSectors], s_cand[kSelSectors], s_above[kSelSectors], s_band[kSelSectors];
  __shared__ int s_count[3][32];
  const SelectTask T = tasks[blockIdx.x];
  const int tid = threadIdx.x;
  const int ns = T.s1 - T.s0;
  const bool listed = ns <= kSelSectors;
  // the sectors' tables, then their values, in shared memory
  int total = 0;
  if (listed) {
    for (int s = tid; s < ns; s += kSelThreads) {
      s_sig[s] = secs[T.s0 + s].sigma;
      s_k[s] = secs[T.s0 + s].k;
    }
    __syncthreads();
    for (int s = 0; s < ns; ++s) total += s_k[s];
    if (total <= kSelValues) {
      int o = 0;
      for (int s = 0; s < ns; ++s) {
        const double* g = s_sig[s];
        for (int j = tid; j < s_k[s]; j += kSelThreads) s_val[o + j] = g[j];
        o += s_k[s];
      }
      __syncthreads();
      if (tid == 0)
        for (int s = 0, q = 0; s < ns; q += s_k[s], ++s) s_sig[s] = s_val + q;
      __syncthreads();
    }
  }
  // 2^p - 1 thresholds a round of the search, as many as give every (sector, threshold) a thread
  int p = 5;
  while (p > 1 && ns << p > kSelThreads) --p;
  if (tid < 32) s_count[0][tid] = 0;      // before the barriers of the sums below
  auto sector = [&](int s) { return listed ? SelectSector{s_sig[s], s_k[s]} : secs[T.s0 + s]; };
  // |sigma|^2 and sigma_max
  double part = 0.0, vmax = 0.0;
  for (int s = 0; s < ns; ++s) {
    const SelectSector S = sector(s);
    for (int j = tid; j < S.k; j += kSelThreads) part = fma(S.sigma[j], S.sigma[j], part);
    if (S.k > 0) vmax = fmax(vmax, S.sigma[0]);
  }
  const double total2 = block_sum(part, dred);
  SelectResult R;
  R.norm_all = sqrt(total2);
  R.band = 0;
  R.pad = 0;
  if (!(total2 > 0.0)) {
    if (tid == 0) {
      R.norm_kept = 0.0; R.trunc_err = 1.0; R.n_candidates = 0; R.status = -1; R.cut = 0.0;
      res[blockIdx.x] = R;
    }
    for (int s = tid; s < ns; s += kSelThreads) kept[T.s0 + s] = 0;
    return;
  }
  double thr = T.cutoff * R.norm_all;
  if (thr == 0.0) thr = 0.0;      // -0.0 has the lowest bits of all
  long long nc_part = 0;
  for (int s = tid; s < ns; s += kSelThreads) {
    const SelectSector S = sector(s);
    const int c = count_gt(S.sigma, S.k, thr);
    if (listed) s_cand[s] = c;
    kept[T.s0 + s] = c;
    nc_part += c;
  }
  const long long nc = block_sum(nc_part, ired);
  int band_total = 0;
  if (nc > T.chi) {
    // v, the largest x with #{sigma >= x} >= chi, is the chi-th largest candidate
    long long lo = thr >= 0.0 ? bits(thr) + 1 : 0, hi = bits(vmax) + 1;      // #{>= lo} >= chi > #{>= hi}
    const int g = p == 1 ? 0 : p, j = tid & ((1 << g) - 1);      // thresholds sit in neighbouring lanes
    for (int r = 0; hi - lo > 1; r = r == 2 ? 0 : r + 1) {
      const long long step = max(1LL, (hi - lo) >> p), x = lo + step * (j + 1);
      const bool tried = j + 1 < 1 << p && x < hi;
      int c = 0;
      if (tried)
        for (int t = tid; t < ns << g; t += kSelThreads) {
          const SelectSector S = sector(t >> g);
          c += count_from(S.sigma, S.k, x);
        }
      for (int o = 1 << g; o < 32; o <<= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
      if ((tid & 31) < 1 << g && c) atomicAdd(&s_count[r][j], c);
      if (tid < 32) s_count[r == 2 ? 0 : r + 1][tid] = 0;      // last read two barriers ago
      __syncthreads();
      const unsigned enough =
          __ballot_sync(0xffffffffu, (tid & 31) < 1 << g && tried && s_count[r][j] >= T.chi);
      const int above = enough ? 32 - __clz(enough) : 0;      // the thresholds that still have chi values
      if (lo + step * (above + 1) < hi && above + 1 < 1 << p) hi = lo + step * (above + 1);
      lo += step * above;
    }
    const double v = __longlong_as_double(lo);
    const double delta = kTieRel * vmax;
    const double upper = v + delta, lower = v - delta;
    long long above_part = 0, band_part = 0;
    for (int s = tid; s < ns; s += kSelThreads) {
      const SelectSector S = sector(s);
      const int cand = listed ? s_cand[s] : count_gt(S.sigma, S.k, thr);
      const int above = count_gt(S.sigma, S.k, upper);
      const int inband = min(count_ge(S.sigma, S.k, lower), cand) - above;
      if (listed) {
        s_above[s] = above;
        s_band[s] = inband;
        s_cand[s] = above + inband;      // from here on: the number kept
      }
      kept[T.s0 + s] = above + inband;
      above_part += above;
      band_part += inband;
    }
    const long long above_total = block_sum(above_part, ired);
    band_total = (int)block_sum(band_part, ired);
    if (tid == 0 && band_total > T.chi - above_total) {      // more ties than places: in sector order
      long long left = T.chi - above_total;
      for (int s = 0; s < ns; ++s) {
        int above, inband;
        if (listed) {
          above = s_above[s];
          inband = s_band[s];
        } else {
          const SelectSector S = secs[T.s0 + s];
          above = count_gt(S.sigma, S.k, upper);
          inband = kept[T.s0 + s] - above;
        }
        const long long take = min((long long)inband, left);
        if (listed) s_cand[s] = above + (int)take;
        kept[T.s0 + s] = above + (int)take;
        left -= take;
      }
    }
    __syncthreads();
  }
  __syncthreads();
  // kept and discarded weight
  double kp = 0.0, dp = 0.0;
  for (int s = 0; s < ns; ++s) {
    const SelectSector S = sector(s);
    const int k = listed ? s_cand[s] : kept[T.s0 + s];
    for (int j = tid; j < S.k; j += kSelThreads) {
      const double w = S.sigma[j] * S.sigma[j];
      if (j < k) kp += w; else dp += w;
    }
  }
  const double kept2 = block_sum(kp, dred);
  const double disc2 = block_sum(dp, dred);
  // the cut: smallest kept value (fixed-order reduction: min is order independent anyway)
  double cmin = 1.0e308;
  for (int s = tid; s < ns; s += kSelThreads) {
    const int k = listed ? s_cand[s] : kept[T.s0 + s];
    if (k > 0) cmin = fmin(cmin, sector(s).sigma[k - 1]);
  }
  for (int o = 16; o; o >>= 1) cmin = fmin(cmin, __shfl_xor_sync(0xffffffffu, cmin, o));
  if ((tid & 31) == 0) dred[tid >> 5] = cmin;
  __syncthreads();
  if (tid == 0) {
    for (int x = 1; x < kSelThreads / 32; ++x) cmin = fmin(cmin, dred[x]);
    R.cut = cmin >= 1.0e308 ? 0.0 : cmin;
    R.norm_kept = sqrt(kept2);
    R.trunc_err = disc2 / total2;
    R.band = band_total;
    R.n_candidates = (int)nc;
    R.status = 0;
    res[blockIdx.x] = R;
  }
}

}  // namespace

cudaError_t launch_select(const SelectSector* d_secs, const SelectTask* d_tasks, int n_tasks,
                          int* d_kept, SelectResult* d_res, cudaStream_t st) {
  if (n_tasks <= 0) return cudaSuccess;
  count_launch();
  select_kernel<<<n_tasks, kSelThreads, 0, st>>>(d_secs, d_tasks, d_kept, d_res);
  return cudaGetLastError();
}

}  // namespace mps
