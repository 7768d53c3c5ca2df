// kernels_update.cu -- the Update step of GenCD (Algorithm 3) on sm_103a.
//
//  * k_update_flat: z += delta_j X_j for accepted columns that may share rows
//    (Thread-Greedy, Greedy), FP64 atomic adds into z (the paper's OpenMP
//    `atomic`, Section 4.2), work spread evenly over the non-zeros of all
//    accepted columns; w_j += delta_j where the column is accepted, or in
//    k_apply_list.
//  * k_shotgun_step: Propose and the Update of w and z for Shotgun's list.
//  * k_refresh_flat: u_i = l'(y_i, z_i) on the rows of the accepted columns,
//    launched after every atomic add of the iteration has landed.
//  * k_coloring_iter: one Coloring iteration fused into a single pass: the
//    columns of one colour class share no row (Section 4.1), so each warp
//    proposes its column and then writes z and u of its own rows with plain
//    stores -- no atomics, no second pass.
//  * k_update_refresh: both passes over a short list in one launch.
//  * k_w_segments, k_fit_segments: z = Xw from the columns with w_j != 0
//    (a warm start is sparse); k_csr_spmv: z = Xw by rows, for a dense w.
//  * k_fill_u: u from z for all rows.
#include <algorithm>

#include "device_math.cuh"
#include "gencd_internal.cuh"

namespace gencd {

template <typename U>
__global__ void __launch_bounds__(kThreads)
    k_fill_u(const double* __restrict__ y, const double* __restrict__ z, int64_t n, int loss,
             const double* __restrict__ tab, U* __restrict__ u, unsigned long long* counts,
             unsigned long long* report) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  const int64_t i0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  for (int64_t i = i0; i < n; i += stride) u[i] = u_value<U>(loss, y[i], z[i], tab);
  if (report && i0 < 2) {  // z = Xw's counts to the host's copy, and reset for the next call
    report[i0] = counts[i0];
    counts[i0] = 0ull;
  }
}

// The applied columns of a list (J[e] >= 0 and D[e] != 0) are laid end to end
// in a virtual range [0, total), and threads take equal parts of that range: a
// 50,000-nnz column is spread over the whole GPU instead of one CTA.
// Whoever applies the list writes list[e] = the column's length | kApplied, or
// 0 for an entry that is not applied; the passes over the range prefix-sum it.

// w_j += delta_j for the applied entries (distinct columns), and list[e]
__global__ void k_apply_list(const int64_t* __restrict__ col_ptr, const int32_t* __restrict__ J,
                             const double* __restrict__ D, int64_t m, double* __restrict__ w,
                             float* __restrict__ w32, uint32_t* __restrict__ list) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < m; e += stride) {
    const int32_t j = J[e];
    const double d = D[e];
    uint32_t l = 0;
    if (j >= 0 && d != 0.0) l = apply_column(j, d, col_ptr, w, w32);
    list[e] = l;
  }
}

// A list of more than kListScanMax entries: lengths without the flag (list[m]
// = 0) for the prefix sum in memory, and the counters
__global__ void k_list_lengths(uint32_t* __restrict__ list, int64_t m, unsigned long long* __restrict__ counters) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  unsigned long long upd = 0, work = 0;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e <= m; e += stride) {
    const uint32_t v = e < m ? list[e] : 0u;
    list[e] = v & ~kApplied;
    upd += v >> 31;
    work += v & ~kApplied;
  }
  upd = warp_sum(upd);
  work = warp_sum(work);
  if ((threadIdx.x & 31) == 0 && upd) {
    atomicAdd(counters + 0, upd);
    atomicAdd(counters + 1, work);
  }
}

// last entry e in [0, m) with off[e] <= q
__device__ __forceinline__ int64_t entry_of(const uint32_t* off, int64_t m, uint32_t q) {
  int64_t lo = 0, hi = m - 1;
  while (lo < hi) {
    const int64_t mid = (lo + hi + 1) >> 1;
    if (off[mid] <= q)
      lo = mid;
    else
      hi = mid - 1;
  }
  return lo;
}

constexpr int kListThreads = 512;

// The offsets of a list's applied columns, off[0..m].  SCAN (m <=
// kListScanMax): every CTA sums the list itself, in shared memory, where the
// searches of its threads then run: 4 KB of L2 reads for 1,024 entries.  On 512
// accepted columns (20,000 non-zeros) the passes over z and u take 4.0 and 4.3
// us; with a launch of its own for the offsets (4.8 us) and searches of nine
// dependent loads in memory they took 4.4 and 6.6.  counters (not null): CTA 0 adds the updates and
// the non-zeros to them.  Not SCAN: the offsets are in memory already.
template <bool SCAN>
__device__ __forceinline__ const uint32_t* list_offsets(const uint32_t* list, int64_t m,
                                                        uint32_t* s_off, unsigned long long* counters) {
  if (!SCAN) return list;
  __shared__ uint32_t s_warp[kListThreads / 32];
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, mi = (int)m;
  uint32_t upd = 0;
  for (int e = tid; e < mi; e += kListThreads) {
    const uint32_t v = list[e];
    upd += v >> 31;
    s_off[e] = v & ~kApplied;
  }
  __syncthreads();
  const int per = (mi + kListThreads - 1) / kListThreads;
  const int e0 = min(tid * per, mi), e1 = min(e0 + per, mi);
  uint32_t mine = 0;
  for (int e = e0; e < e1; ++e) mine += s_off[e];
  uint32_t incl = mine;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, incl, d);
    if (lane >= d) incl += y;
  }
  if (lane == 31) s_warp[wid] = incl;
  __syncthreads();
  uint32_t run = incl - mine, total = 0;
#pragma unroll
  for (int v = 0; v < kListThreads / 32; ++v) {
    if (v < wid) run += s_warp[v];
    total += s_warp[v];
  }
  for (int e = e0; e < e1; ++e) {
    const uint32_t x = s_off[e];
    s_off[e] = run;
    run += x;
  }
  if (tid == 0) s_off[mi] = total;
  if (counters && blockIdx.x == 0) {
    upd = warp_sum(upd);
    if (lane == 0 && upd) atomicAdd(counters + 0, (unsigned long long)upd);
    if (tid == 0 && total) atomicAdd(counters + 1, (unsigned long long)total);
  }
  __syncthreads();
  return s_off;
}

// z_i += delta_j X_ij over the applied columns (atomic: columns may share rows).
// A thread takes one position at a time, or four consecutive ones with one
// search when there are more than threads; with the accepted columns short
// that is all latency, with millions of non-zeros the FP64 atomics.  1,024
// columns of up to 50,000 non-zeros on 2e8 take 150 us a pass, 490 with a
// search per position and half of the threads.
template <typename V, bool SCAN>
__global__ void __launch_bounds__(kListThreads)
    k_update_flat(const int64_t* __restrict__ col_ptr, const int32_t* __restrict__ row_idx,
                  const V* __restrict__ val, const int32_t* J, const double* D, const uint32_t* list, int64_t m,
                  double* z, unsigned long long* counters) {
  __shared__ uint32_t s_off[SCAN ? kListScanMax + 1 : 1];
  pdl_trigger();
  pdl_wait();
  const uint32_t* off = list_offsets<SCAN>(list, m, s_off, counters);
  const int64_t total = off[m], threads = (int64_t)gridDim.x * kListThreads;
  const int run = total > threads ? 4 : 1;
  for (int64_t q0 = ((int64_t)blockIdx.x * kListThreads + threadIdx.x) * run; q0 < total; q0 += threads * run) {
    int64_t e = entry_of(off, m, (uint32_t)q0), end = off[e + 1], at = col_ptr[J[e]] - off[e];
    double d = D[e];
#pragma unroll 1
    for (int64_t q = q0; q < q0 + run && q < total; ++q) {
      if (q >= end) {  // the next applied column
        do end = off[++e + 1];
        while (q >= end);
        at = col_ptr[J[e]] - off[e];
        d = D[e];
      }
      atomicAdd(z + row_idx[at + q], d * (double)val[at + q]);
    }
  }
}

// u_i = l'(y_i, z_i) on the rows of the applied columns, or on all rows when
// the iteration touched at least n entries (one dense pass is cheaper then).
// Neighbouring warps of the range lie on different SMs: in FP64 the logistic
// derivative takes some 12 FP64 operations, which an SM starts about two a
// cycle, so few rows have to be spread over all of them (100,000 rows: 7.8 us,
// 9.5 with neighbouring warps in one CTA; ncu).
template <typename U, bool SCAN>
__global__ void __launch_bounds__(kListThreads)
    k_refresh_flat(const int64_t* __restrict__ col_ptr, const int32_t* __restrict__ row_idx,
                   const int32_t* J, const uint32_t* list, int64_t m, const double* __restrict__ y, const double* z,
                   int64_t n, int loss, const double* __restrict__ tab, U* u, unsigned long long* counters) {
  __shared__ uint32_t s_off[SCAN ? kListScanMax + 1 : 1];
  pdl_trigger();
  pdl_wait();
  const uint32_t* off = list_offsets<SCAN>(list, m, s_off, counters);
  const int64_t total = off[m], stride = (int64_t)gridDim.x * kListThreads;
  const int64_t q0 = ((int64_t)(threadIdx.x >> 5) * gridDim.x + blockIdx.x) * 32 + (threadIdx.x & 31);
  if (total >= n) {
    for (int64_t i = q0; i < n; i += stride) u[i] = u_value<U>(loss, y[i], z[i], tab);
    return;
  }
  for (int64_t q = q0; q < total; q += stride) {
    const int64_t e = entry_of(off, m, (uint32_t)q);
    const int32_t i = row_idx[col_ptr[J[e]] + ((uint32_t)q - off[e])];
    u[i] = u_value<U>(loss, y[i], z[i], tab);
  }
}

// Both passes over a short list in one launch: the CTAs are one cluster, whose
// barrier stands between the last addition into z and the first u.  Every launch
// of an iteration of little work costs 2 us or more, on the device and on the
// host; kClusterCtas SMs refresh up to short_list() non-zeros in about that time.
constexpr int kClusterCtas = 8;

template <typename V, typename U>
__global__ void __launch_bounds__(kListThreads)
    k_update_refresh(const int64_t* __restrict__ col_ptr, const int32_t* __restrict__ row_idx,
                     const V* __restrict__ val, const int32_t* J, const double* D, const uint32_t* list, int64_t m,
                     const double* __restrict__ y, double* z, int64_t n, int loss, const double* __restrict__ tab,
                     U* u, unsigned long long* counters) {
  __shared__ uint32_t s_off[kListScanMax + 1];
  pdl_trigger();
  pdl_wait();
  const uint32_t* off = list_offsets<true>(list, m, s_off, counters);
  const int64_t total = off[m], threads = (int64_t)kClusterCtas * kListThreads;
  // neighbouring warps on different SMs, as in k_refresh_flat
  const int64_t q0 = ((int64_t)(threadIdx.x >> 5) * kClusterCtas + blockIdx.x) * 32 + (threadIdx.x & 31);
  for (int64_t q = q0; q < total; q += threads) {
    const int64_t e = entry_of(off, m, (uint32_t)q);
    const int64_t p = col_ptr[J[e]] + ((uint32_t)q - off[e]);
    atomicAdd(z + row_idx[p], D[e] * (double)val[p]);
  }
  asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
  if (total >= n) {
    for (int64_t i = q0; i < n; i += threads) u[i] = u_value<U>(loss, y[i], load_l2(z + i), tab);
    return;
  }
  for (int64_t q = q0; q < total; q += threads) {
    const int64_t e = entry_of(off, m, (uint32_t)q);
    const int32_t i = row_idx[col_ptr[J[e]] + ((uint32_t)q - off[e])];
    u[i] = u_value<U>(loss, y[i], load_l2(z + i), tab);
  }
}

// Shotgun's Propose, Accept (all of J) and the Update of w and z in one pass:
// a proposal reads u and its own w_j only, so its column's step goes into z at
// once (u follows when all have landed: k_refresh_flat).  A CTA takes `per`
// <= 8 columns, one a warp; a column of more than kWarpColumn entries is left
// to the whole CTA.
//
// Bound: latency (dependent loads, then the FP64 step), so every column has
// its own warp at once and long ones 256 threads: this takes 13 us on 800
// columns of 1 to 5,000 non-zeros (FP32); one warp a column took 32, with a
// launch each for the list's plan (4.4) and z (5.2) after it.  The step is evaluated by one thread: a warp's
// FP64 instruction holds the pipe for some 16 cycles an SM.
constexpr int kWarpColumn = 256;
constexpr int kShotgunCols = kThreads / 32;

template <typename V, typename U>
__global__ void __launch_bounds__(kThreads)
    k_shotgun_step(const int64_t* __restrict__ col_ptr, const int32_t* __restrict__ row_idx,
                   const V* __restrict__ val, const U* u, const double* __restrict__ bjs,
                   const double* __restrict__ ib, const int32_t* J, int64_t m, int per, int early, double n, double lam,
                   double* w, float* w32, double* z, uint32_t* list, unsigned long long* counters) {
  __shared__ int64_t s_long[kShotgunCols];
  __shared__ int s_nlong;
  __shared__ uint32_t s_len[kShotgunCols];
  __shared__ double s_sum[kThreads / 32], s_d;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  if (!early) pdl_wait();  // J is the output of an earlier kernel, which may still run
  pdl_trigger();
  if (tid == 0) s_nlong = 0;
  if (lane == 0) s_len[wid] = 0u;
  __syncthreads();
  const int64_t first = (int64_t)blockIdx.x * per;
  const bool mine = wid < per && first + wid < m;  // this warp's column
  int32_t wj = 0, r0 = 0;
  int64_t ws = 0;
  uint32_t wlen = 0;
  V v0 = V(0);
  if (mine) {  // its extent and first entries, which no iteration writes
    wj = J[first + wid];
    ws = col_ptr[wj];
    wlen = (uint32_t)(col_ptr[wj + 1] - ws);
    if ((uint32_t)lane < wlen) {
      r0 = row_idx[ws + lane];
      v0 = val[ws + lane];
    }
  }
  if (early) pdl_wait();
  auto step = [&](int64_t e, int32_t j, double sum) {  // one thread: the column's step, applied to w
    double d, f;
    eq7_step(sum / n, w[j], lam, bjs[j], ib[j], d, f);
    list[e] = d != 0.0 ? apply_column(j, d, col_ptr, w, w32) : 0u;
    return d;
  };
  if (mine) {
    const int64_t e = first + wid, s = ws;
    const int32_t j = wj;
    const uint32_t len = wlen;
    if (lane == 0) s_len[wid] = len;
    if (len > (uint32_t)kWarpColumn) {
      if (lane == 0) s_long[atomicAdd(&s_nlong, 1)] = e;
    } else {
      V acc = (uint32_t)lane < len ? v0 * (V)u[r0] : V(0);
#pragma unroll 4
      for (uint32_t t = lane + 32; t < len; t += 32) acc = fma(val[s + t], (V)u[row_idx[s + t]], acc);
      const double sum = warp_sum((double)acc);
      double d = 0.0;
      if (lane == 0) d = step(e, j, sum);
      d = __shfl_sync(0xffffffffu, d, 0);
      if (d != 0.0) {
        if ((uint32_t)lane < len) atomicAdd(z + r0, d * (double)v0);
#pragma unroll 4
        for (uint32_t t = lane + 32; t < len; t += 32) atomicAdd(z + row_idx[s + t], d * (double)val[s + t]);
      }
    }
  }
  __syncthreads();
  const int nlong = s_nlong;
  for (int q = 0; q < nlong; ++q) {  // uniform across the CTA
    const int64_t e = s_long[q];
    const int32_t j = J[e];
    const int64_t s = col_ptr[j];
    const uint32_t len = (uint32_t)(col_ptr[j + 1] - s);
    V acc = V(0);
#pragma unroll 4
    for (uint32_t t = tid; t < len; t += kThreads) acc = fma(val[s + t], (V)u[row_idx[s + t]], acc);
    const double part = warp_sum((double)acc);
    if (lane == 0) s_sum[wid] = part;
    __syncthreads();
    if (tid == 0) {
      double sum = 0.0;
      for (int v = 0; v < kThreads / 32; ++v) sum += s_sum[v];
      s_d = step(e, j, sum);
    }
    __syncthreads();
    const double d = s_d;
    if (d != 0.0) {
#pragma unroll 4
      for (uint32_t t = tid; t < len; t += kThreads) atomicAdd(z + row_idx[s + t], d * (double)val[s + t]);
    }
  }
  if (tid == 0) {  // the non-zeros proposed on
    unsigned long long work = 0;
    for (int v = 0; v < kShotgunCols; ++v) work += s_len[v];
    if (work) atomicAdd(counters + 1, work);
  }
}

// One warp per column of the colour class.
//
// Bound: latency, a chain of ten dependent loads and FP64 operations, at one
// launch per iteration.  So the class is spread thinly (a warp's FP64
// instruction holds the pipe for some 16 cycles an SM), and what no iteration
// writes (the class, the columns' extents, first entries and their y) is read
// while the previous iteration still runs: 3.6 us an iteration on classes of
// about 70 columns (FP64), 6.9 with eight warps a CTA and a plain launch.
template <typename V, typename U>
__global__ void __launch_bounds__(kThreads)
    k_coloring_iter(const int64_t* __restrict__ col_ptr, const int32_t* __restrict__ row_idx,
                    const V* __restrict__ val, U* u, double* w, float* w32, const double* __restrict__ bjs,
                    const double* __restrict__ ib, double* z, const double* __restrict__ y, const int32_t* perm,
                    int64_t q, const int32_t* __restrict__ color_ptr, const int32_t* __restrict__ cols_by_color,
                    double n, double lam, int loss, const double* __restrict__ tab, int early,
                    unsigned long long* counters) {
  const int lane = threadIdx.x & 31;
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  bool waited = !early;
  if (!early) pdl_wait();  // perm is the output of an earlier kernel, which may still run
  pdl_trigger();
  const int32_t colour = perm[q];
  const int32_t lo = color_ptr[colour], hi = color_ptr[colour + 1];
  unsigned long long upd = 0, work = 0;
  for (int64_t e = lo + warp; e < hi; e += nwarps) {
    const int32_t j = cols_by_color[e];
    const int64_t s = col_ptr[j], t = col_ptr[j + 1];
    const bool have = s + lane < t;
    const int32_t i0 = have ? row_idx[s + lane] : 0;
    const V v0 = have ? val[s + lane] : V(0);
    const double y0 = have ? y[i0] : 0.0;
    if (!waited) {
      pdl_wait();
      waited = true;
    }
    const double z0 = have ? z[i0] : 0.0;  // no other column of the class has row i0
    V acc = have ? v0 * (V)u[i0] : V(0);
    for (int64_t p = s + lane + 32; p < t; p += 32) acc = fma(val[p], (V)u[row_idx[p]], acc);
    const double g = warp_sum((double)acc) / n;
    const double wj = w[j];
    double d, f;
    eq7_step(g, wj, lam, bjs[j], ib[j], d, f);  // identical on every lane
    work += (unsigned long long)(t - s);
    if (d != 0.0) {
      // every lane has read its u values above (warp_sum synchronised them)
      if (have) {
        const double zi = z0 + d * (double)v0;
        z[i0] = zi;
        u[i0] = u_value<U>(loss, y0, zi, tab);
      }
      for (int64_t p = s + lane + 32; p < t; p += 32) {
        const int32_t i = row_idx[p];
        const double zi = z[i] + d * (double)val[p];
        z[i] = zi;
        u[i] = u_value<U>(loss, y[i], zi, tab);
      }
      if (lane == 0) {
        w[j] = wj + d;
        if (w32) w32[j] = w_mirror(wj + d);
      }
      upd += 1;
      work += (unsigned long long)(t - s);
    }
  }
  if (!waited) pdl_wait();
  if (lane == 0 && (upd | work)) {
    atomicAdd(counters + 0, upd);
    atomicAdd(counters + 1, work);
  }
}

// rows of X x, a warp each
template <typename V>
__device__ __forceinline__ void sum_rows(const int64_t* __restrict__ row_ptr, const int32_t* __restrict__ col_idx,
                                         const V* __restrict__ csr_val, const double* __restrict__ x, int64_t n,
                                         double* __restrict__ out) {
  const int lane = threadIdx.x & 31;
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t i = warp; i < n; i += nwarps) {
    double acc = 0.0;
    for (int64_t q = row_ptr[i] + lane; q < row_ptr[i + 1]; q += 32)
      acc = fma((double)csr_val[q], x[col_idx[q]], acc);
    acc = warp_sum(acc);
    if (lane == 0) out[i] = acc;
  }
}

template <typename V>
__global__ void __launch_bounds__(kThreads)
    k_csr_spmv(const int64_t* __restrict__ row_ptr, const int32_t* __restrict__ col_idx,
               const V* __restrict__ csr_val, const double* __restrict__ x, int64_t n, double* __restrict__ out) {
  sum_rows(row_ptr, col_idx, csr_val, x, n, out);
}

__global__ void k_mirror_w(const double* __restrict__ w, int64_t k, float* __restrict__ w32) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < k; j += stride) w32[j] = w_mirror(w[j]);
}

// z = X w from the columns with w_j != 0, in segments of kSegEntries
// non-zeros so that a long column is spread over many warps.  Pass 1 lists the
// segments (writes the float copy of w and zeroes z): a CTA counts its columns'
// segments, takes their place in the list with one atomic add, and also sums
// the listed non-zeros into *total.  The list holds list_cap(k, nnz) segments,
// those of all columns.
__global__ void __launch_bounds__(kThreads)
    k_w_segments(const double* __restrict__ w, float* __restrict__ w32, const int64_t* __restrict__ col_ptr, int64_t k,
                 int32_t* __restrict__ seg_j, uint32_t* __restrict__ seg_t,
                 unsigned long long* __restrict__ count, unsigned long long* __restrict__ total, int64_t n,
                 double* __restrict__ z) {
  constexpr int PER = 4;
  __shared__ uint32_t s_warp[kThreads / 32];
  __shared__ unsigned long long s_base;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  for (int64_t i = (int64_t)blockIdx.x * kThreads + threadIdx.x; i < n; i += (int64_t)gridDim.x * kThreads) z[i] = 0.0;
  for (int64_t base = (int64_t)blockIdx.x * (PER * kThreads); base < k;
       base += (int64_t)gridDim.x * (PER * kThreads)) {  // uniform across the CTA
    uint32_t nseg[PER], mine = 0;
    unsigned long long len_sum = 0;
#pragma unroll
    for (int q = 0; q < PER; ++q) {
      const int64_t j = base + q * kThreads + threadIdx.x;
      nseg[q] = 0;
      if (j >= k) continue;
      const double wj = w[j];
      if (w32) w32[j] = w_mirror(wj);
      if (wj != 0.0) {  // NaN counts as non-zero
        const int64_t len = col_ptr[j + 1] - col_ptr[j];
        nseg[q] = (uint32_t)((len + kSegEntries - 1) / kSegEntries);
        len_sum += (unsigned long long)len;
      }
      mine += nseg[q];
    }
    uint32_t incl = mine;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, incl, d);
      if (lane >= d) incl += y;
    }
    len_sum = warp_sum(len_sum);
    if (lane == 0 && len_sum) atomicAdd(total, len_sum);
    if (lane == 31) s_warp[wid] = incl;
    __syncthreads();
    uint32_t before = 0, all = 0;
    for (int v = 0; v < kThreads / 32; ++v) {
      if (v < wid) before += s_warp[v];
      all += s_warp[v];
    }
    if (threadIdx.x == 0) s_base = all ? atomicAdd(count, (unsigned long long)all) : 0ull;
    __syncthreads();
    uint64_t pos = s_base + before + (incl - mine);
#pragma unroll
    for (int q = 0; q < PER; ++q)
      for (uint32_t t = 0; t < nseg[q]; ++t, ++pos) {
        seg_j[pos] = (int32_t)(base + q * kThreads + threadIdx.x);
        seg_t[pos] = t;
      }
    __syncthreads();  // s_warp and s_base are reused
  }
}

// pass 2: a warp per segment adds w_j X_ij into z (FP64 atomics).  When the listed
// non-zeros exceed `limit`: z by rows if the row-major copy is there (row_ptr not
// null), else nothing
template <typename V>
__global__ void __launch_bounds__(kThreads)
    k_fit_segments(const int32_t* __restrict__ seg_j, const uint32_t* __restrict__ seg_t,
                   const unsigned long long* __restrict__ count, const unsigned long long* __restrict__ total,
                   unsigned long long limit, const int64_t* __restrict__ col_ptr, const int32_t* __restrict__ row_idx,
                   const V* __restrict__ val, const double* __restrict__ w, const int64_t* __restrict__ row_ptr,
                   const int32_t* __restrict__ col_idx, const V* __restrict__ csr_val, int64_t n,
                   double* __restrict__ z) {
  const int64_t m = (int64_t)*count;
  if (*total > limit) {
    if (row_ptr) sum_rows(row_ptr, col_idx, csr_val, w, n, z);
    return;
  }
  const int lane = threadIdx.x & 31;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t g = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; g < m; g += nwarps) {
    const int32_t j = seg_j[g];
    const double wj = w[j];
    const int64_t s = col_ptr[j] + (int64_t)seg_t[g] * kSegEntries, e0 = col_ptr[j + 1];
    const int64_t e = s + kSegEntries < e0 ? s + kSegEntries : e0;
#pragma unroll 4
    for (int64_t t = s + lane; t < e; t += 32) atomicAdd(z + row_idx[t], wj * (double)val[t]);
  }
}

// ---------------------------------------------------------------------------
// launchers

// Improve delta_j (Algorithm 3; Section 4.1: further steps of the quadratic
// approximation per accepted increment): one warp per accepted column j
// repeats the Eq. 7 step on coordinate j from w_j + d, with g_j at
// z + d X_j (the iteration-start z: every accepted increment is improved
// before any is applied), until a step is 0 or `steps` steps.  FP64 in both
// storage modes.
template <typename V>
__global__ void k_improve_list(const int32_t* __restrict__ J, double* __restrict__ D, int64_t m,
                               const int64_t* __restrict__ col_ptr, const int32_t* __restrict__ row_idx,
                               const V* __restrict__ val, const double* __restrict__ y, const double* __restrict__ z,
                               const double* __restrict__ w, const double* __restrict__ bjs,
                               const double* __restrict__ ibs, int loss, double lam, double inv_n, int steps) {
  const int lane = threadIdx.x & 31;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t e = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; e < m; e += nw) {
    const int32_t j = J[e];
    if (j < 0) continue;
    const double bj = bjs[j];
    if (!(bj > 0.0)) continue;  // a column without entries: its step is already exact
    const double wj = w[j], ibj = ibs[j];
    const int64_t a = col_ptr[j], b = col_ptr[j + 1];
    double d = D[e];
    for (int s = 0; s < steps; ++s) {  // warp-uniform: g is the same in every lane
      double acc = 0.0;
      for (int64_t t = a + lane; t < b; t += 32) {
        const double x = (double)val[t];
        const int32_t i = row_idx[t];
        acc += x * loss_deriv(loss, y[i], z[i] + d * x);
      }
      const double g = warp_sum(acc) * inv_n;
      double step, phi;
      eq7_step(g, wj + d, lam, bj, ibj, step, phi);
      if (step == 0.0) break;
      d += step;
    }
    if (lane == 0) D[e] = d;
  }
}

int launch_improve_list(gencd_problem* p, const int32_t* J, double* D, int64_t m) {
  const int steps = p->params.improve_steps;
  if (steps <= 0 || m <= 0) return GENCD_OK;
  const int grid = grid_for(m * 32, kThreads, p->num_sms * 8);
  const double inv_n = 1.0 / (double)p->n;
  if (p->precision == GENCD_F64)
    k_improve_list<double><<<grid, kThreads, 0, p->stream>>>(J, D, m, p->col_ptr, p->row_idx, (const double*)p->val,
                                                             p->y, p->z, p->w, p->bj, p->ib, p->loss, p->lambda,
                                                             inv_n, steps);
  else
    k_improve_list<float><<<grid, kThreads, 0, p->stream>>>(J, D, m, p->col_ptr, p->row_idx, (const float*)p->val,
                                                            p->y, p->z, p->w, p->bj, p->ib, p->loss, p->lambda, inv_n,
                                                            steps);
  p->prof.launches[K_UPDATE] += 1;
  GENCD_CUDA_TRY(cudaGetLastError());
  return GENCD_OK;
}

int launch_fill_u(gencd_problem* p, unsigned long long* counts, unsigned long long* report) {
  if (p->n == 0) return GENCD_OK;
  const int grid = grid_for(p->n, kThreads, p->num_sms * 8);
  if (p->precision == GENCD_F64)
    k_fill_u<double><<<grid, kThreads, 0, p->stream>>>(p->y, p->z, p->n, p->loss, p->ltab, (double*)p->u, counts, report);
  else
    k_fill_u<float><<<grid, kThreads, 0, p->stream>>>(p->y, p->z, p->n, p->loss, p->ltab, (float*)p->u, counts, report);
  p->prof.launches[K_SETUP] += 1;
  GENCD_CUDA_TRY(cudaGetLastError());
  return GENCD_OK;
}

int launch_fill_u64(gencd_problem* p) {
  k_fill_u<double><<<grid_for(p->n, kThreads, p->num_sms * 8), kThreads, 0, p->stream>>>(
      p->y, p->z, p->n, p->loss, p->ltab, p->u64, nullptr, nullptr);
  p->prof.launches[K_SETUP] += 1;
  GENCD_CUDA_TRY(cudaGetLastError());
  return GENCD_OK;
}

// w and list_off for the accepted entries of the list (J, d)
int launch_apply_list(gencd_problem* p, const int32_t* J, const double* d, int64_t m) {
  if (m <= 0) return GENCD_OK;
  k_apply_list<<<grid_for(m, kThreads, p->num_sms * 8), kThreads, 0, p->stream>>>(p->col_ptr, J, d, m, p->w, p->w32,
                                                                                  p->list_off);
  p->prof.launches[K_UPDATE] += 1;
  GENCD_CUDA_TRY(cudaGetLastError());
  return GENCD_OK;
}

// a long list's offsets, in list_off, and its counts
static int prefix_long_list(gencd_problem* p, int64_t m) {
  unsigned long long* ctr = reinterpret_cast<unsigned long long*>(p->dscal + 4);
  k_list_lengths<<<grid_for(m + 1, kThreads, p->num_sms * 8), kThreads, 0, p->stream>>>(p->list_off, m, ctr);
  p->prof.launches[K_UPDATE] += 1;
  GENCD_CUDA_TRY(cudaGetLastError());
  return exclusive_scan(p, p->list_off, p->list_off, m + 1, p->scan_tmp);
}

// CTAs of the passes over a list: as many threads as are resident
static int list_grid(const gencd_problem* p) { return p->num_sms * 4; }

// Non-zeros up to which a list's two passes go in one launch (k_update_refresh).
// Twenty Thread-Greedy iterations on uniform columns, in one launch / in two:
// FP64 2,000 non-zeros a list 638 / 669 us, 320 518 / 577; FP32 3,840 non-zeros
// 522 / 557, 320 431 / 478; beyond, eight SMs are too few: 18,000 to 19,000 FP32
// non-zeros 678 to 697 / 525 to 529.
static int64_t short_list(const gencd_problem* p) { return p->precision == GENCD_F64 ? 4096 : 8192; }

// Update (Algorithm 3) of z for the list (J, d) whose w has been applied
// (list_off), the counters, and u
int launch_update_refresh(gencd_problem* p, const int32_t* J, const double* d, int64_t m) {
  if (m <= 0) return GENCD_OK;
  unsigned long long* ctr = reinterpret_cast<unsigned long long*>(p->dscal + 4);
  if (m <= kListScanMax && m * p->max_len <= short_list(p)) {
    cudaEvent_t ev = nullptr;
    prof_begin(p, K_UPDATE, &ev);
    auto go = [&](auto kernel, auto* val, auto* u) {
      return launch_cluster_overlapped(kernel, kClusterCtas, dim3(kClusterCtas), dim3(kListThreads), 0, launch_on(p),
                                       p->col_ptr, p->row_idx, val, J, d, p->list_off, m, p->y, p->z, p->n, p->loss,
                                       p->ltab, u, ctr);
    };
    const cudaError_t err = p->precision == GENCD_F64
                                ? go(k_update_refresh<double, double>, (const double*)p->val, (double*)p->u)
                                : go(k_update_refresh<float, float>, (const float*)p->val, (float*)p->u);
    prof_end(p, ev);
    GENCD_CUDA_TRY(err);
    return GENCD_OK;
  }
  const bool scan = m <= kListScanMax;
  if (!scan) GENCD_TRY(prefix_long_list(p, m));
  cudaEvent_t ev = nullptr;
  prof_begin(p, K_UPDATE, &ev);
  auto go = [&](auto kernel, auto* val) {
    return launch_overlapped(kernel, list_grid(p), kListThreads, 0, launch_on(p), p->col_ptr, p->row_idx, val, J, d,
                             p->list_off, m, p->z, ctr);
  };
  cudaError_t err;
  if (p->precision == GENCD_F64)
    err = go(scan ? k_update_flat<double, true> : k_update_flat<double, false>, (const double*)p->val);
  else
    err = go(scan ? k_update_flat<float, true> : k_update_flat<float, false>, (const float*)p->val);
  prof_end(p, ev);
  GENCD_CUDA_TRY(err);
  return launch_refresh_list(p, J, m, true);
}

// u on the rows of the list's applied columns, after z.  counted: the list's
// counts are in the counters already (launch_update_refresh); else (Shotgun's
// fused step) they are added here.
int launch_refresh_list(gencd_problem* p, const int32_t* J, int64_t m, bool counted) {
  if (m <= 0) return GENCD_OK;
  unsigned long long* ctr = counted ? nullptr : reinterpret_cast<unsigned long long*>(p->dscal + 4);
  const bool scan = m <= kListScanMax;
  if (!scan && !counted) GENCD_TRY(prefix_long_list(p, m));
  cudaEvent_t ev = nullptr;
  prof_begin(p, K_REFRESH, &ev);
  auto go = [&](auto kernel, auto* u) {
    return launch_overlapped(kernel, list_grid(p), kListThreads, 0, launch_on(p), p->col_ptr, p->row_idx, J, p->list_off,
                             m, p->y, p->z, p->n, p->loss, p->ltab, u, ctr);
  };
  cudaError_t err;
  if (p->precision == GENCD_F64)
    err = go(scan ? k_refresh_flat<double, true> : k_refresh_flat<double, false>, (double*)p->u);
  else
    err = go(scan ? k_refresh_flat<float, true> : k_refresh_flat<float, false>, (float*)p->u);
  prof_end(p, ev);
  GENCD_CUDA_TRY(err);
  return GENCD_OK;
}

// Shotgun's iteration on the list J up to z: propose, accept all, w and z.
// early: no kernel still running may be writing J.
int launch_shotgun_step(gencd_problem* p, const int32_t* J, int64_t m, bool early) {
  if (m <= 0) return GENCD_OK;
  unsigned long long* ctr = reinterpret_cast<unsigned long long*>(p->dscal + 4);
  // two CTAs per SM before a CTA takes a second column
  const int per = (int)std::min<int64_t>(kShotgunCols, (m + 2 * p->num_sms - 1) / (2 * p->num_sms));
  const unsigned grid = (unsigned)((m + per - 1) / per);
  cudaEvent_t ev = nullptr;
  prof_begin(p, K_PROPOSE_LIST, &ev);
  cudaError_t err;
  if (p->precision == GENCD_F64)
    err = launch_overlapped(k_shotgun_step<double, double>, grid, kThreads, 0, launch_on(p), p->col_ptr, p->row_idx,
                            (const double*)p->val, (const double*)p->u, p->bj, p->ib, J, m, per, early ? 1 : 0,
                            (double)p->n, p->lambda, p->w, p->w32, p->z, p->list_off, ctr);
  else
    err = launch_overlapped(k_shotgun_step<float, float>, grid, kThreads, 0, launch_on(p), p->col_ptr, p->row_idx,
                            (const float*)p->val, (const float*)p->u, p->bj, p->ib, J, m, per, early ? 1 : 0,
                            (double)p->n, p->lambda, p->w, p->w32, p->z, p->list_off, ctr);
  prof_end(p, ev);
  GENCD_CUDA_TRY(err);
  return GENCD_OK;
}

// early: no kernel still running may be writing the permutation
int launch_coloring_iter(gencd_problem* p, int64_t q, bool early) {
  const int64_t warps = p->max_class > 0 ? p->max_class : 1;
  // two warps per SM before a CTA takes a second one
  const int per = (int)std::min<int64_t>(kThreads / 32, (warps + 2 * p->num_sms - 1) / (2 * p->num_sms));
  const int grid = grid_for(warps, per, p->num_sms * 8);
  unsigned long long* ctr = reinterpret_cast<unsigned long long*>(p->dscal + 4);
  cudaEvent_t ev = nullptr;
  prof_begin(p, K_COLOR_ITER, &ev);
  cudaError_t err;
  if (p->precision == GENCD_F64)
    err = launch_overlapped(k_coloring_iter<double, double>, grid, 32 * per, 0, launch_on(p), p->col_ptr, p->row_idx,
                            (const double*)p->val, (double*)p->u, p->w, p->w32, p->bj, p->ib, p->z, p->y, p->perm, q,
                            p->color_ptr, p->cols_by_color, (double)p->n, p->lambda, p->loss, p->ltab, early ? 1 : 0, ctr);
  else
    err = launch_overlapped(k_coloring_iter<float, float>, grid, 32 * per, 0, launch_on(p), p->col_ptr, p->row_idx,
                            (const float*)p->val, (float*)p->u, p->w, p->w32, p->bj, p->ib, p->z, p->y, p->perm, q,
                            p->color_ptr, p->cols_by_color, (double)p->n, p->lambda, p->loss, p->ltab, early ? 1 : 0, ctr);
  prof_end(p, ev);
  GENCD_CUDA_TRY(err);
  return GENCD_OK;
}

// z = Xw, u = l'(y, z) and (FP32 mode) the float copy of w, from the
// coefficients in p->w.
//
// Sparse coefficients: their columns are scattered into z, which reads no more
// of X than those columns and needs no row-major copy (whose build sorts every
// non-zero).  Otherwise the rows are summed: once the row-major copy is there,
// the second launch takes one or the other by the listed non-zeros; before that
// the host does, after a wait (finish_state_from_w), and builds it.  The line is
// drawn at 2/5 of the non-zeros: a call took, by columns with w_j != 0, scattered
// / by rows, on 4.0e7 FP32 non-zeros 48 / 276 us at 0.5%, 84 / 276 at 12.5%, 155 /
// 276 at 40%, 309 / 276 at 100%, and on 2.0e7 FP64 non-zeros 52 / 123, 74 / 123,
// 116 / 123 and 164 / 123 us.  The listing costs a dense w 6 to 8 us (284 and 128
// us in all, 13 us on a million columns of 3 non-zeros).
//
// At most kFitRowsNnz non-zeros: always by rows.  Reading all of X takes no
// longer there than listing w's segments, and the sums have a fixed order, so
// that equal problems get equal z to the last bit (the scatter's atomic adds
// do not).
static int state_by_rows(gencd_problem* p) {
  GENCD_TRY(build_csr(p));
  GENCD_TRY(launch_csr_spmv(p, p->w, p->z));
  return launch_fill_u(p);
}

// non-zeros of the listed columns up to which they are scattered
static unsigned long long fit_limit(const gencd_problem* p) { return (unsigned long long)(p->nnz / 5 * 2); }

int launch_state_from_w(gencd_problem* p) {
  p->fit_open = false;
  if (p->nnz <= kFitRowsNnz) {
    if (p->w32) {
      k_mirror_w<<<grid_for(p->k, kThreads, p->num_sms * 8), kThreads, 0, p->stream>>>(p->w, p->k, p->w32);
      p->prof.launches[K_SETUP] += 1;
      GENCD_CUDA_TRY(cudaGetLastError());
    }
    return state_by_rows(p);
  }
  unsigned long long* total = reinterpret_cast<unsigned long long*>(p->dscal + kScalFit);  // zero between calls
  unsigned long long* count = total + 1;
  unsigned long long* host = reinterpret_cast<unsigned long long*>(p->hpin + kScalFit);
  const unsigned long long limit = fit_limit(p);
  const int g = p->num_sms * 8;
  k_w_segments<<<grid_for(std::max((p->k + 3) / 4, p->n), kThreads, g), kThreads, 0, p->stream>>>(
      p->w, p->w32, p->col_ptr, p->k, p->list_j, p->list_off, count, total, p->n, p->z);
  if (p->precision == GENCD_F64)
    k_fit_segments<double><<<g, kThreads, 0, p->stream>>>(p->list_j, p->list_off, count, total, limit, p->col_ptr,
                                                          p->row_idx, (const double*)p->val, p->w, p->row_ptr,
                                                          p->col_idx, (const double*)p->csr_val, p->n, p->z);
  else
    k_fit_segments<float><<<g, kThreads, 0, p->stream>>>(p->list_j, p->list_off, count, total, limit, p->col_ptr,
                                                         p->row_idx, (const float*)p->val, p->w, p->row_ptr,
                                                         p->col_idx, (const float*)p->csr_val, p->n, p->z);
  p->prof.launches[K_SETUP] += 2;
  GENCD_CUDA_TRY(cudaGetLastError());
  GENCD_TRY(launch_fill_u(p, total, host));
  p->fit_open = p->row_ptr == nullptr;
  return GENCD_OK;
}

int finish_state_from_w(gencd_problem* p) {
  if (!p->fit_open) return 0;
  p->fit_open = false;
  if (reinterpret_cast<const unsigned long long*>(p->hpin + kScalFit)[0] <= fit_limit(p)) return 0;
  GENCD_TRY(state_by_rows(p));
  return 1;
}

int launch_csr_spmv(gencd_problem* p, const double* x, double* out) {
  if (p->n == 0) return GENCD_OK;
  const int grid = grid_for(p->n * 32, kThreads, p->num_sms * 8);
  if (p->precision == GENCD_F64)
    k_csr_spmv<double><<<grid, kThreads, 0, p->stream>>>(p->row_ptr, p->col_idx, (const double*)p->csr_val,
                                                         x, p->n, out);
  else
    k_csr_spmv<float><<<grid, kThreads, 0, p->stream>>>(p->row_ptr, p->col_idx, (const float*)p->csr_val,
                                                        x, p->n, out);
  p->prof.launches[K_SETUP] += 1;
  GENCD_CUDA_TRY(cudaGetLastError());
  return GENCD_OK;
}

}  // namespace gencd
