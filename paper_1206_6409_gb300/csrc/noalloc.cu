// noalloc.cu -- gencd_propose_all_noalloc: the streaming Propose over all
// columns for callers that cannot allocate device memory.
//
// Who needs it: a host thread that must not synchronise the device (cudaMalloc
// and cudaFree can wait for the GPU to go idle), a process whose framework
// has already reserved all device memory in its own pool, or code that
// enqueues work while another thread captures the stream into a graph.  Such
// a caller passes the inputs and outputs; the call creates no problem handle
// and allocates nothing.  Its scratch (per-column sums, the tile map and u) is
// a file-scope device array of fixed size that every GPU loading this library
// holds until the process exits.
//
// The scratch is shared by every call on a device and keeps the last call's
// contents: each call clears the part it accumulates into before using it,
// and two calls that overlap on the GPU (different streams, no ordering
// between them) race on it.
#include <algorithm>
#include <mutex>
#include <string>

#include "device_math.cuh"
#include "gencd_internal.cuh"

namespace gencd {

constexpr int64_t kNoAllocMaxCols = int64_t(1) << 19;  // columns (k)
constexpr int kNoAllocItems = 8;                        // nnz per lane
constexpr int64_t kNoAllocTile = 32 * kNoAllocItems;
constexpr int64_t kNoAllocMaxNnz = int64_t(1) << 25;   // non-zeros
constexpr int64_t kNoAllocMaxTiles = kNoAllocMaxNnz / kNoAllocTile;
constexpr int64_t kNoAllocMaxURows = int64_t(1) << 19;  // rows whose u fits the scratch

// layout: [0, K) column sums X_j^T u, [K, 2K) sums of X_ij^2, the tile map
// (int32, max tiles + 1 entries), then u; 2 K + (max tiles + 2) / 2 + rows =
// 1,638,401 doubles = 13,107,208 bytes (13.1 MB, 12.5 MiB)
constexpr int64_t kNoAllocTileMapAt = 2 * kNoAllocMaxCols;
constexpr int64_t kNoAllocUAt = kNoAllocTileMapAt + (kNoAllocMaxTiles + 2) / 2;
static __device__ __align__(256) double g_noalloc_scratch[kNoAllocUAt + kNoAllocMaxURows];

// What each call prepares, in one launch: the sums and the KKT maximum
// cleared, the tile map, and (u not null) u_i = l'(y_i, z_i)
__global__ void __launch_bounds__(kThreads)
    k_na_prep(const int64_t* __restrict__ col_ptr, int64_t k, int64_t ntiles, int32_t* __restrict__ tile_col,
              double* __restrict__ sums, double* __restrict__ kkt, const double* __restrict__ y,
              const double* __restrict__ z, int64_t n, int loss, double* __restrict__ u) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  const int64_t i0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  for (int64_t j = i0; j < k; j += stride) {
    sums[j] = 0.0;
    sums[k + j] = 0.0;
    const int64_t s = col_ptr[j], e = col_ptr[j + 1];
    for (int64_t t = (s + kNoAllocTile - 1) / kNoAllocTile; t * kNoAllocTile < e; ++t) tile_col[t] = (int32_t)j;
  }
  if (u)
    for (int64_t i = i0; i < n; i += stride) u[i] = loss_deriv(loss, y[i], z[i]);
  if (i0 == 0) {
    tile_col[ntiles] = (int32_t)(k - 1);
    *kkt = 0.0;
  }
}

__device__ __forceinline__ void na_emit(double* __restrict__ sums, int64_t k, int32_t c, double su, double sq,
                                        bool whole) {
  if (whole) {
    sums[c] = su;
    sums[k + c] = sq;
  } else {
    atomicAdd(sums + c, su);
    atomicAdd(sums + k + c, sq);
  }
}

// Lane-segmented pass over the non-zeros: the sums X_j^T u and, with them, the
// sums of squares that give beta_j without a separate pass.  A warp owns a
// tile of 256 entries, a lane 8 of them; a column inside one lane is stored, a
// column cut by lanes is summed across the warp, and only a tile's first and
// last columns are added atomically.  U_ARRAY: u from the scratch, else
// evaluated per non-zero.  vec: the caller's arrays are 16-byte aligned (they
// need no padding: a tile's tail takes scalar loads).
//
// Bound: the FP64 pipe (about 2 multiply-adds a cycle and SM): the two sums
// take 2 operations per non-zero (21 us on 6.0e6 non-zeros, whose 72 MB take
// 11).  This takes 48 us there; evaluating the logistic u per non-zero (an
// exponential and a division, some 50 operations) instead of once per row
// (10 us with the rest of k_na_prep) took 620.
template <bool U_ARRAY>
__global__ void __launch_bounds__(kThreads, 3)
    k_na_stream(const int64_t* __restrict__ col_ptr, const int32_t* __restrict__ row_idx,
                const double* __restrict__ val, const double* __restrict__ y, const double* __restrict__ z,
                const double* __restrict__ u, int loss, const int32_t* __restrict__ tile_col, int64_t nnz,
                int64_t ntiles, int64_t k, int vec, double* __restrict__ sums) {
  constexpr int N = kNoAllocItems;
  const unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t t = warp; t < ntiles; t += nwarps) {  // warp-uniform
    const int64_t a = t * kNoAllocTile + (int64_t)lane * N;
    const int m = a >= nnz ? 0 : (nnz - a < N ? (int)(nnz - a) : N);  // entries of this lane
    int32_t r[N];
    double v[N], uu[N];
    if (vec && m == N) {
#pragma unroll
      for (int q = 0; q < N / 4; ++q) {
        const int4 x = __ldcs(reinterpret_cast<const int4*>(row_idx + a) + q);
        r[4 * q] = x.x, r[4 * q + 1] = x.y, r[4 * q + 2] = x.z, r[4 * q + 3] = x.w;
      }
#pragma unroll
      for (int q = 0; q < N / 2; ++q) {
        const double2 x = __ldcs(reinterpret_cast<const double2*>(val + a) + q);
        v[2 * q] = x.x, v[2 * q + 1] = x.y;
      }
    } else {
#pragma unroll
      for (int i = 0; i < N; ++i) {
        r[i] = i < m ? row_idx[a + i] : 0;
        v[i] = i < m ? val[a + i] : 0.0;
      }
    }
#pragma unroll
    for (int i = 0; i < N; ++i) {
      if (U_ARRAY)
        uu[i] = i < m ? __ldg(u + r[i]) : 0.0;
      else
        uu[i] = i < m ? loss_deriv(loss, y[r[i]], z[r[i]]) : 0.0;
    }
    // the lane's runs: `cont` is what continues a column from the left, `tail`
    // the last run if its column started in this lane
    double cu = 0.0, cq = 0.0, tu = 0.0, tq = 0.0;
    bool has_tail = false;
    int32_t c = 0;
    int64_t cend = 0;
    const int64_t tile_end = (t + 1) * kNoAllocTile < nnz ? (t + 1) * kNoAllocTile : nnz;
    if (m > 0) {
      int32_t lo = tile_col[t], hi = tile_col[t + 1];  // column holding position a
      while (lo < hi) {
        const int32_t mid = (lo + hi + 1) >> 1;
        if (col_ptr[mid] <= a)
          lo = mid;
        else
          hi = mid - 1;
      }
      c = lo;
      cend = col_ptr[c + 1];
      bool mine = col_ptr[c] >= a;  // the current run's column started in this lane
      double su = 0.0, sq = 0.0;
#pragma unroll
      for (int i = 0; i < N; ++i) {
        if (i < m) {
          while (a + i >= cend) {  // column c ended before this entry
            if (mine) {
              na_emit(sums, k, c, su, sq, true);
            } else {
              cu = su;
              cq = sq;
            }
            ++c;
            cend = col_ptr[c + 1];
            su = sq = 0.0;
            mine = true;
          }
          su = fma(v[i], uu[i], su);
          sq = fma(v[i], v[i], sq);
        }
      }
      if (mine) {
        tu = su;
        tq = sq;
        has_tail = true;
      } else {
        cu = su;
        cq = sq;
      }
    }
    // columns cut by lanes: T_L = the parts of the column that lane L continues
    const bool stop = m == 0 || has_tail;
    bool ended;
    lane_suffix_sum2(cu, cq, stop, lane, ended);
    const double nu = __shfl_down_sync(FULL, cu, 1), nq = __shfl_down_sync(FULL, cq, 1);
    // lane 0's continued column began in an earlier tile
    const int32_t c0 = tile_col[t];
    if (lane == 0 && col_ptr[c0] < a) na_emit(sums, k, c0, cu, cq, false);
    if (has_tail)
      na_emit(sums, k, c, lane < 31 ? tu + nu : tu, lane < 31 ? tq + nq : tq, cend <= tile_end);
  }
}

// Steps, proxies and the KKT maximum.  A column with w_j = 0 and |g_j| <=
// lambda does not move; the others are queued in shared memory and taken
// packed, since each costs two more FP64 divisions (11.5 us on k = 150,000,
// 18.4 with every column evaluated in place).
__global__ void __launch_bounds__(kThreads)
    k_na_finalize(const double* __restrict__ sums, const double* __restrict__ w, int64_t k, double n, double lam,
                  double beta, int beta_mode, double* __restrict__ delta, double* __restrict__ phi,
                  double* __restrict__ kkt) {
  constexpr int PER = 4;
  __shared__ int s_n;
  __shared__ int32_t s_j[PER * kThreads];
  __shared__ double s_g[PER * kThreads];
  double vmax = 0.0;
  for (int64_t base = (int64_t)blockIdx.x * (PER * kThreads); base < k;
       base += (int64_t)gridDim.x * (PER * kThreads)) {  // uniform across the CTA
    if (threadIdx.x == 0) s_n = 0;
    __syncthreads();
#pragma unroll
    for (int q = 0; q < PER; ++q) {
      const int64_t j = base + q * kThreads + threadIdx.x;
      if (j >= k) continue;
      const double g = sums[j] / n;
      // a sum of squares beyond the type's range takes the general steps
      const bool finite_sq = isfinite(sums[k + j]);
      if (w[j] == 0.0 && fabs(g) <= lam && finite_sq) {
        delta[j] = 0.0;
        phi[j] = 0.0;
      } else {
        const int slot = atomicAdd(&s_n, 1);
        s_j[slot] = (int32_t)j;
        s_g[slot] = g;
      }
    }
    __syncthreads();
    const int na = s_n;
    for (int e = threadIdx.x; e < na; e += kThreads) {
      const int64_t j = s_j[e];
      const double g = s_g[e], wj = w[j];
      const double bj = beta_mode ? beta : beta * (sums[k + j] / n);
      double d, f;
      eq7_step(g, wj, lam, bj, bj > 0.0 ? 1.0 / bj : 0.0, d, f);
      delta[j] = d;
      phi[j] = f;
      const double v = kkt_violation(g, wj, lam);
      vmax = (v > vmax || v != v) ? v : vmax;
    }
    __syncthreads();  // the queue is reused
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const double x = __shfl_xor_sync(0xffffffffu, vmax, o);
    vmax = (x > vmax || x != x) ? x : vmax;
  }
  if ((threadIdx.x & 31) == 0) atomic_max_nonneg(kkt, vmax);
}

// device address of the scratch array, looked up once per device with that
// device current (the host symbol is not a device address)
static std::mutex g_na_mutex;
static double* g_na_ptr[64] = {nullptr};

static int noalloc_scratch(double** out) {
  int dev = 0;
  GENCD_CUDA_TRY(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64) return fail_plan("device index out of range for the no-allocation scratch table");
  std::lock_guard<std::mutex> lock(g_na_mutex);
  if (!g_na_ptr[dev]) {
    void* ptr = nullptr;
    GENCD_CUDA_TRY(cudaGetSymbolAddress(&ptr, g_noalloc_scratch));
    g_na_ptr[dev] = static_cast<double*>(ptr);
  }
  *out = g_na_ptr[dev];
  return GENCD_OK;
}

}  // namespace gencd

using namespace gencd;

extern "C" int gencd_propose_all_noalloc(int64_t n, int64_t k, int64_t nnz, const int64_t* col_ptr,
                                         const int32_t* row_idx, const double* val, const double* y,
                                         const double* z, const double* w, int32_t loss, double lambda,
                                         int32_t beta_mode, double* delta, double* phi, double* kkt,
                                         void* stream) try {
  set_error("");
  if (n < 1 || k < 1 || nnz < 0) return fail_plan("need n >= 1, k >= 1, nnz >= 0");
  if (k > kNoAllocMaxCols || nnz > kNoAllocMaxNnz)
    return fail_plan(("gencd_propose_all_noalloc handles at most " + std::to_string(kNoAllocMaxCols) +
                      " columns and " + std::to_string(kNoAllocMaxNnz) + " non-zeros (its scratch is a fixed "
                      "device array); use a problem handle for larger inputs")
                         .c_str());
  if (!col_ptr || !y || !z || !w || !delta || !phi || !kkt || (nnz > 0 && (!row_idx || !val)))
    return fail_plan("a required pointer is NULL");
  if (loss != GENCD_LOSS_SQUARED && loss != GENCD_LOSS_LOGISTIC) return fail_plan("unknown loss");
  if (!(lambda >= 0.0) || !std::isfinite(lambda) || (beta_mode != 0 && beta_mode != 1))
    return fail_plan("lambda must be finite and >= 0, beta_mode 0 or 1");
  double* scratch = nullptr;
  GENCD_TRY(noalloc_scratch(&scratch));
  double* sums = scratch;
  int32_t* tile_col = reinterpret_cast<int32_t*>(scratch + kNoAllocTileMapAt);
  cudaStream_t st = (cudaStream_t)stream;
  int sms = 0, dev = 0;
  GENCD_CUDA_TRY(cudaGetDevice(&dev));
  GENCD_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  const int g = sms * 8;
  const int64_t ntiles = (nnz + kNoAllocTile - 1) / kNoAllocTile;
  // u once per row when it fits the scratch and no row goes unused on
  // average (n <= nnz); else per non-zero
  double* u = n <= kNoAllocMaxURows && n <= nnz ? scratch + kNoAllocUAt : nullptr;
  const int vec = (((uintptr_t)row_idx | (uintptr_t)val) & 15u) == 0 ? 1 : 0;
  k_na_prep<<<grid_for(u ? std::max(k, n) : k, kThreads, g), kThreads, 0, st>>>(col_ptr, k, ntiles, tile_col, sums, kkt,
                                                                               y, z, n, loss, u);
  if (ntiles > 0) {
    const int gs = grid_for(ntiles * 32, kThreads, sms * 3);  // resident CTAs
    if (u)
      k_na_stream<true><<<gs, kThreads, 0, st>>>(col_ptr, row_idx, val, y, z, u, loss, tile_col, nnz, ntiles, k, vec,
                                                 sums);
    else
      k_na_stream<false><<<gs, kThreads, 0, st>>>(col_ptr, row_idx, val, y, z, u, loss, tile_col, nnz, ntiles, k, vec,
                                                  sums);
  }
  const double beta = loss == GENCD_LOSS_SQUARED ? 1.0 : 0.25;
  k_na_finalize<<<grid_for((k + 3) / 4, kThreads, g), kThreads, 0, st>>>(sums, w, k, (double)n, lambda, beta, beta_mode,
                                                                       delta, phi, kkt);
  GENCD_CUDA_TRY(cudaGetLastError());
  return GENCD_OK;
}
GENCD_CATCH
