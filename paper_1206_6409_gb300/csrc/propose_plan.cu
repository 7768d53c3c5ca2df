// propose_plan.cu -- row-slab layout of the streaming propose (g = X^T u over
// all columns) on sm_103a.
//
// Gathering u_i at random rows costs one 32-byte L2 sector per 4- or 8-byte
// value, which makes a plain CSC pass L2-bound long before HBM is saturated.
// Here the rows are cut into slabs of at most 192 KB of u.  A persistent CTA
// (one per SM, 1024 threads) copies the u slab of its work into shared memory
// once and gathers from there.  Every (slab, column) "pair" (entries regrouped
// slab by slab, with 16-bit in-slab rows) produces one partial sum, added
// atomically into the column's g_j.  Columns that would produce about two
// partials per non-zero or more ("light", when there are many: the rule is in
// build_plan_impl) keep a compact CSC copy and the lane-segmented pass with
// gathers from L2.
//
// Within a slab the kernel works like the CSC pass: a warp owns a tile of
// consecutive entries, a lane 8 (FP32) or 16 (FP64) of them (128-bit loads of
// rows and values), a lane sums its entries pair by pair in registers and adds each
// run's sum into g_j (an atomic add that returns nothing: other slabs and
// tiles add to the same column); a run cut by lane boundaries is combined by
// a segmented warp suffix sum first, and a full tile inside one pair is
// reduced by the warp.  Sums are kept in the storage precision (FP32 atomics
// in FP32 mode), so the order of a heavy column's additions, and with it the
// last bits of g_j, can differ between launches.
#include <cuda_bf16.h>

#include <algorithm>
#include <type_traits>
#include <vector>

#include "device_math.cuh"
#include "gencd_internal.cuh"

namespace gencd {

constexpr int kSlabBytes = 192 * 1024;
// Entries of a slab are stored in tiles of kSlabTile, in the order in which a
// warp's lanes load them: a lane owns 16 consecutive entries (or 8, taking half
// a tile at a time), and its v-th 16-byte vector lies next to the other lanes'
// v-th ones, so a load of a warp is one contiguous 512 bytes with 16 entries a
// lane and two runs of 256 with 8 (slab_at, load_lane).
constexpr int kSlabTile = 512;
// Shape of the row-slab kernel: threads, tiles of loads in flight beyond the
// current one, entries per lane.  FP32 is bound by instructions and loads in
// flight: 1024 / 1 / 8 takes 83 us with the light columns on 4e7 non-zeros,
// 768 / 1 / 16 92 and 512 / 1 / 16 112.  FP64 is bound by its pipe, and a lane's
// 16 entries halve the additions that combine the lanes: 10 Thread-Greedy
// iterations on 2e7 non-zeros take 1259 us with 768 / 0 / 16, 1284 with 512 / 1 /
// 16, 1322 with 1024 / 0 / 8.  768 threads leave 80 registers each, which the FP64
// kernel exceeds by 14 words (56 bytes spilled a thread); with a tile in flight
// it would spill more.
constexpr int kSlabThreadsF32 = 1024;
constexpr int kSlabThreadsF64 = 768;
constexpr int kSlabDepthF32 = 1;
constexpr int kSlabDepthF64 = 0;
constexpr int kSlabItemsF32 = 8;
constexpr int kSlabItemsF64 = 16;
constexpr int kSlabPad = kSlabTile;  // slabs are padded to whole tiles
constexpr int kSlabZeroSlot = 4;   // shared u slots past the slab (16 B); the first holds 0

// ---------------------------------------------------------------------------
// the kernel

// N values as 16-byte vectors, `step` values from one vector to the next
template <typename V, int N>
__device__ __forceinline__ void load_vals(const V* __restrict__ p, V (&v)[N], int step) {
  constexpr int PER = 16 / (int)sizeof(V);  // values per 128-bit load
#pragma unroll
  for (int q = 0; q < N / PER; ++q) {
    if (sizeof(V) == 4) {
      const float4 x = __ldcs(reinterpret_cast<const float4*>(p + q * step));
      v[4 * q] = (V)x.x, v[4 * q + 1] = (V)x.y, v[4 * q + 2] = (V)x.z, v[4 * q + 3] = (V)x.w;
    } else {
      const double2 x = __ldcs(reinterpret_cast<const double2*>(p + q * step));
      v[2 * q] = (V)x.x, v[2 * q + 1] = (V)x.y;
    }
  }
}

template <typename G>
__device__ __forceinline__ void emit_pair(G* out, uint32_t slot, G s, bool whole) {
  if (whole)
    out[slot] = s;
  else
    atomicAdd(out + slot, s);
}

// Values of a lane's entries as stored by the plan (SV): float or double,
// bfloat16 (kept packed, two per register, widened on use), or none at all
// (NoVal: index-only columns, every value 1; the column scale is applied to
// the column's sum outside the streaming loop).
struct NoVal {};

// a heavy column's run sum into g_j: other slabs and tiles add to the same
// column, so always atomically (index-only storage: the sum of u over the
// column's rows; who reads g_j applies the column's value)
template <typename G>
__device__ __forceinline__ void add_col(G* gacc, uint32_t j, G v) {
  atomicAdd(gacc + j, v);
}

template <typename SV, int N>
struct ValRegs;

template <int N>
struct ValRegs<float, N> {
  float v[N];
  __device__ __forceinline__ void load(const float* __restrict__ p, int step = 4) { load_vals<float, N>(p, v, step); }
  __device__ __forceinline__ float get(int i) const { return v[i]; }
};

template <int N>
struct ValRegs<double, N> {
  double v[N];
  __device__ __forceinline__ void load(const double* __restrict__ p, int step = 2) { load_vals<double, N>(p, v, step); }
  __device__ __forceinline__ double get(int i) const { return v[i]; }
};

template <int N>
struct ValRegs<__nv_bfloat16, N> {
  uint32_t w[N / 2];  // value 2q in the low half of w[q], 2q + 1 in the high half
  __device__ __forceinline__ void load(const __nv_bfloat16* __restrict__ p, int step = 8) {
#pragma unroll
    for (int q = 0; q < N / 8; ++q) {
      const uint4 x = __ldcs(reinterpret_cast<const uint4*>(p + q * step));
      w[4 * q] = x.x, w[4 * q + 1] = x.y, w[4 * q + 2] = x.z, w[4 * q + 3] = x.w;
    }
  }
  __device__ __forceinline__ float get(int i) const {  // bfloat16 -> float: the upper 16 bits
    const uint32_t x = w[i >> 1];
    return __uint_as_float((i & 1) ? (x & 0xffff0000u) : (x << 16));
  }
};

template <int N>
struct ValRegs<NoVal, N> {
  __device__ __forceinline__ void load(const NoVal*, int = 0) {}
  __device__ __forceinline__ float get(int) const { return 1.0f; }
};

// values per 16-byte vector of a stored value (index-only storage has none)
template <typename SV>
__host__ __device__ constexpr int vector_of() {
  return std::is_same<SV, NoVal>::value ? 8 : 16 / (int)sizeof(SV);
}

// where entry x of a tile (x < kSlabTile, in pair order) is stored, in vectors of
// VW elements
template <int VW>
__device__ __forceinline__ uint32_t slab_at(uint32_t x) {
  const uint32_t owner = x >> 4, i = x & 15u;
  return (i / VW) * (32 * VW) + owner * VW + i % VW;
}

// the entries of one lane: ITEMS in-slab rows (128-bit loads of 8) and values
template <typename SV, int ITEMS>
struct LaneLoad {
  uint4 rr[ITEMS / 8];
  ValRegs<SV, ITEMS> val;
};

// a0: the first entry, in pair order, of the warp's 32 * ITEMS ones
template <typename SV, int ITEMS>
__device__ __forceinline__ void load_lane(const uint16_t* __restrict__ s_row, const SV* __restrict__ s_val,
                                          uint32_t a0, int lane, LaneLoad<SV, ITEMS>& L) {
  constexpr int VW = vector_of<SV>();
  const uint32_t tile = a0 & ~(uint32_t)(kSlabTile - 1);
  const uint32_t owner = ITEMS == 16 ? (uint32_t)lane : ((a0 >> 8) & 1u) * 16u + ((uint32_t)lane >> 1);
  const uint32_t half = ITEMS == 16 ? 0u : (uint32_t)lane & 1u;  // which 8 of the owner's 16 entries
#pragma unroll
  for (int h = 0; h < ITEMS / 8; ++h)
    L.rr[h] = __ldcs(reinterpret_cast<const uint4*>(s_row + tile + (half + h) * 256u + owner * 8u));
  L.val.load(s_val + tile + half * (8 / VW) * (32 * VW) + owner * VW, 32 * VW);
}

// start bits of a lane's ITEMS entries (one byte per 8 entries, little-endian)
template <int ITEMS>
__device__ __forceinline__ uint32_t lane_mask(const uint8_t* __restrict__ pmask, uint32_t a) {
  if (ITEMS == 16) return reinterpret_cast<const uint16_t*>(pmask)[a >> 4];
  return pmask[a >> 3];
}

// Segmented suffix sum over the lanes: T_L = x_L + x_{L+1} + ... + x_M where M
// is the first lane >= L whose bit is set in `stops` (all lanes to 31 when there
// is none).  M is known from the ballot, so a step is one shuffle and one
// addition; in FP64, whose additions are what the passes wait for, only as many
// steps as the longest run of the warp takes.
template <typename V>
__device__ __forceinline__ V lane_suffix_sum(V x, uint32_t stops, int lane) {
  const uint32_t from = stops >> lane;
  const int last = from ? lane + __ffs(from) - 1 : 31;
  V t = x;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    if (sizeof(V) == 8 && !__any_sync(0xffffffffu, lane + d <= last)) break;
    const V tn = __shfl_down_sync(0xffffffffu, t, d);
    if (lane + d <= last) t += tn;
  }
  return t;
}

// Pairs are numbered in entry order; pmask holds one byte per 8 entries whose
// bit i says "entry 8g + i starts a pair", and tile_pair[t] is the pair of the
// tile's first entry.  A lane finds the pair of its first entry from a warp
// prefix count of the start bits, so no pair table is searched.  Per lane:
// runs that start and end inside the lane are added into g_j as they end; the
// run that continues from the left (cont) and the run that leaves to the right
// (tail) are combined across the warp by a segmented suffix sum, so a pair
// takes one atomic add per tile it touches.
// TileStage: one tile's loads for one lane: ITEMS rows and values, the start
// bits, and the pair of the tile's first entry.
template <typename SV, int ITEMS>
struct TileStage {
  LaneLoad<SV, ITEMS> L;
  uint32_t m, q0;
};

template <typename SV, int ITEMS>
__device__ __forceinline__ void load_stage(const uint16_t* __restrict__ s_row, const SV* __restrict__ s_val,
                                           const uint8_t* __restrict__ pmask,
                                           const uint32_t* __restrict__ tile_pair, int t, int t1, uint32_t base,
                                           int tb, int lane, TileStage<SV, ITEMS>& S) {
  if (t < t1) {
    S.q0 = __ldg(tile_pair + t);
    const uint32_t a0 = base + (uint32_t)(t - tb) * (32 * ITEMS);
    load_lane<SV, ITEMS>(s_row, s_val, a0, lane, S.L);
    S.m = lane_mask<ITEMS>(pmask, a0 + lane * ITEMS);
  }
}

// Barrier of the warps that share a CTA's u slab: the whole CTA (BAR_THREADS
// = 0), or the first BAR_THREADS threads on named barrier 1 when other warps
// of the CTA do other work (the fused pass below).
template <int BAR_THREADS>
__device__ __forceinline__ void slab_barrier() {
  if (BAR_THREADS == 0)
    __syncthreads();
  else
    asm volatile("bar.sync 1, %0;" ::"n"(BAR_THREADS) : "memory");
}

// tiles of one size (32 lanes of 16 or of 8 entries) over the slabs' entries
struct SlabTiles {
  const uint32_t* tile_pair;        // pair holding a tile's first entry
  const int32_t* tile_slab;         // slab of each tile
  const int32_t* slab_tile_begin;   // nslabs + 1
  const int32_t* cta_tile_begin;    // grid + 1
  const uint32_t* slab_off;         // first entry of each slab
};

// The row-slab pass of one CTA's contiguous run of tiles [t0, t_end), by the
// warps warp = 0 .. nw - 1 of the slab group (ITEMS entries per lane, a tile
// is 32 * ITEMS entries; DEPTH tiles of loads in flight per warp beyond the
// one being processed).
template <typename V, typename U, typename G, int DEPTH, int ITEMS, typename SV, int BAR_THREADS>
__device__ __forceinline__ void slab_pass(const uint16_t* __restrict__ s_row, const SV* __restrict__ s_val,
                                          const uint8_t* __restrict__ pmask, const uint32_t* __restrict__ pair_col,
                                          const SlabTiles& T, int t0, const int t_end,
                                          const U* u, int64_t n, int32_t slab_rows,
                                          G* sums, int64_t second, U* s_u, const int warp, const int nw,
                                          const int gtid, const int gthreads) {
  constexpr uint32_t NOT_FIRST = ((1u << ITEMS) - 1u) & ~1u;  // start bits after a lane's first entry
  const unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  if (gtid == 0) s_u[slab_rows] = U(0);  // the row of padding entries (index-only storage)
  bool waited = false;
  while (t0 < t_end) {
    const int r = T.tile_slab[t0];
    const int tb = T.slab_tile_begin[r], t1 = min(t_end, T.slab_tile_begin[r + 1]);
    const uint32_t base = T.slab_off[r];  // the slab's entries
    G* gacc = sums + (r & 1 ? second : 0);
    const int64_t row0 = (int64_t)r * slab_rows;
    const int rows = (int)min((int64_t)slab_rows, n - row0);
    TileStage<SV, ITEMS> stg[DEPTH > 0 ? DEPTH : 1];
    int t = t0 + warp;
#pragma unroll
    for (int d = 0; d < DEPTH; ++d)
      load_stage<SV, ITEMS>(s_row, s_val, pmask, T.tile_pair, t + d * nw, t1, base, tb, lane, stg[d]);
    slab_barrier<BAR_THREADS>();  // the previous slab is no longer read
    if (!waited) {  // the plan is read while the kernel that writes u still runs
      pdl_wait();
      waited = true;
    }
    {  // 16-byte loads, four in flight per thread, when u + row0 is 16-byte aligned
      const bool al = (reinterpret_cast<uintptr_t>(u + row0) & 15u) == 0;
      const int nvec = al ? (int)(((int64_t)rows * (int64_t)sizeof(U)) / 16) : 0;
      const uint4* src = reinterpret_cast<const uint4*>(u + row0);
      uint4* dst = reinterpret_cast<uint4*>(s_u);
      int i0 = gtid;
      for (; i0 + 3 * gthreads < nvec; i0 += 4 * gthreads) {
        uint4 x[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) x[q] = load_l2(src + i0 + q * gthreads);
#pragma unroll
        for (int q = 0; q < 4; ++q) dst[i0 + q * gthreads] = x[q];
      }
      for (; i0 < nvec; i0 += gthreads) dst[i0] = load_l2(src + i0);
      for (int i = (int)((int64_t)nvec * 16 / (int64_t)sizeof(U)) + gtid; i < rows; i += gthreads) s_u[i] = load_l2(u + row0 + i);
    }
    slab_barrier<BAR_THREADS>();
    for (; t < t1; t += nw) {  // warp-uniform loop
      TileStage<SV, ITEMS> cur;
      if (DEPTH > 0) {
        cur = stg[0];
#pragma unroll
        for (int d = 0; d + 1 < DEPTH; ++d) stg[d] = stg[d + 1];
        load_stage<SV, ITEMS>(s_row, s_val, pmask, T.tile_pair, t + DEPTH * nw, t1, base, tb, lane, stg[DEPTH - 1]);
      } else {
        load_stage<SV, ITEMS>(s_row, s_val, pmask, T.tile_pair, t, t1, base, tb, lane, cur);
      }
      const uint32_t q0 = cur.q0, m = cur.m;
      // pair of the lane's first entry: q0 + the tile's start bits after its
      // first entry and up to the lane's
      const uint32_t cnt = __popc(lane == 0 ? (m & NOT_FIRST) : m);
      uint32_t incl = cnt;
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const uint32_t y = __shfl_up_sync(FULL, incl, d);
        if (lane >= d) incl += y;
      }
      uint32_t q = q0 + (incl - cnt) + (lane > 0 ? (m & 1u) : 0u);
      // columns of the pairs this lane may emit, loaded early: the tile's
      // first pair (lane 0) and the pair of the lane's last run
      const bool lead = lane == 0 && !(m & 1u);
      const uint32_t col0 = lead ? __ldg(pair_col + q0) : 0u;
      const uint32_t col_last = m != 0u ? __ldg(pair_col + q + __popc(m & NOT_FIRST)) : 0u;
      V cont = V(0), tail = V(0);
      bool has_tail = false;
      {
        U uu[ITEMS];
#pragma unroll
        for (int h = 0; h < ITEMS / 8; ++h) {
          const uint32_t w4[4] = {cur.L.rr[h].x, cur.L.rr[h].y, cur.L.rr[h].z, cur.L.rr[h].w};
#pragma unroll
          for (int k2 = 0; k2 < 4; ++k2) {
            uu[8 * h + 2 * k2] = s_u[w4[k2] & 0xffffu];
            uu[8 * h + 2 * k2 + 1] = s_u[w4[k2] >> 16];
          }
        }
        // one FMA chain over the lane's entries; at each start bit after
        // entry 0 the running sum closes a run: the first run (continuing
        // from the left, or a whole run when it began at entry 0) or a run
        // between two start bits (whole: stored); the last run stays in acc.
        // Only the latter are a branch: some lane of the warp has a start at
        // almost every i, and a branch there cost all lanes its instructions.
        const uint32_t inner = m & NOT_FIRST;
        const uint32_t earliest = inner & (0u - inner), later = inner ^ earliest;  // the first start bit, the others
        V acc = V(0), first = V(0);
#pragma unroll
        for (int i = 0; i < ITEMS; ++i) {
          if ((later >> i) & 1u)  // a run that started and ended inside the lane
            add_col<G>(gacc, __ldg(pair_col + q + __popc(inner & ((1u << i) - 1u))), (G)acc);
          first = (earliest >> i) & 1u ? acc : first;
          acc = (inner >> i) & 1u ? V(0) : acc;
          acc = fma((V)cur.L.val.get(i), (V)uu[i], acc);
        }
        if (inner) {
          if (m & 1u)
            add_col<G>(gacc, __ldg(pair_col + q), (G)first);  // started at entry 0, ended inside
          else
            cont = first;  // continues from the left
          tail = acc;  // the last run started inside the lane
          has_tail = true;
        } else if (m & 1u) {  // one run, starting at the lane's first entry
          tail = acc;
          has_tail = true;
        } else {
          cont = acc;
        }
      }
      const uint32_t stops = __ballot_sync(FULL, m != 0u);
      if (stops == 0u) {
        // the whole tile lies inside pair q0
        const V sum = warp_sum(cont);
        if (lane == 0) add_col<G>(gacc, col0, (G)sum);
      } else {
        const V tsum = lane_suffix_sum(cont, stops, lane);
        const V t1s = __shfl_down_sync(FULL, tsum, 1);
        if (lead) add_col<G>(gacc, col0, (G)tsum);  // pair from the previous tile
        if (has_tail) add_col<G>(gacc, col_last, (G)(tail + (lane < 31 ? t1s : V(0))));
      }
    }
    t0 = t1;
  }
  if (!waited) pdl_wait();
}

// THREADS per CTA (one CTA per SM); see slab_pass
template <typename V, typename U, typename G, int THREADS, int DEPTH, int ITEMS, typename SV>
__global__ void __launch_bounds__(THREADS, 1)
    k_propose_slabs(const uint16_t* __restrict__ s_row, const SV* __restrict__ s_val,
                    const uint8_t* __restrict__ pmask, const uint32_t* __restrict__ pair_col, SlabTiles T,
                    const U* u, int64_t n, int32_t slab_rows, G* gacc, int64_t second) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  U* s_u = reinterpret_cast<U*>(smem_raw);
  pdl_trigger();
  slab_pass<V, U, G, DEPTH, ITEMS, SV, 0>(s_row, s_val, pmask, pair_col, T, T.cta_tile_begin[blockIdx.x],
                                          T.cta_tile_begin[blockIdx.x + 1], u, n, slab_rows, gacc, second, s_u,
                                          threadIdx.x >> 5, blockDim.x >> 5, threadIdx.x, blockDim.x);
}

// ---------------------------------------------------------------------------
// the light columns: a compact CSC copy streamed in 256-entry tiles, u gathered
// from L2.  Column starts are marked like pair starts above (one byte per 8
// entries), tile_lc[t] is the light column of the tile's first entry, and the
// same per-lane runs / segmented suffix sum assign every partial sum to its
// column without a search; results go to out[light_cols[lc]].
constexpr int kLightItems = 8;
constexpr int kLightTile = 32 * kLightItems;

__device__ __forceinline__ void load_rows8(const int32_t* __restrict__ p, int32_t (&r)[8]) {
  const int4 a = __ldcs(reinterpret_cast<const int4*>(p));
  const int4 b = __ldcs(reinterpret_cast<const int4*>(p) + 1);
  r[0] = a.x, r[1] = a.y, r[2] = a.z, r[3] = a.w, r[4] = b.x, r[5] = b.y, r[6] = b.z, r[7] = b.w;
}

// one lane's loads of a light tile: 8 rows, 8 values (as stored), the start
// bits, and the light column of the tile's first entry
template <typename SV>
struct LightStage {
  int32_t r[8];
  ValRegs<SV, 8> val;
  uint32_t m, lc0;
};

template <typename SV>
__device__ __forceinline__ void load_light_stage(const int32_t* __restrict__ row, const SV* __restrict__ val,
                                                 const uint8_t* __restrict__ lmask,
                                                 const int32_t* __restrict__ tile_lc, int64_t t, int64_t ntiles,
                                                 int64_t nnz, int lane, LightStage<SV>& S) {
  S.m = 0;
  if (t < ntiles) {
    S.lc0 = (uint32_t)__ldg(tile_lc + t);
    const int64_t a = t * kLightTile + (int64_t)lane * kLightItems;
    if (a < nnz) {  // the arrays are padded: a lane's 8 entries are in bounds
      load_rows8(row + a, S.r);
      S.val.load(val + a);
      S.m = lmask[a >> 3];
    }
  }
}

// One light tile's sums from its loads `cur` (index-only columns: the sums of u
// over their rows); results go to out[light_cols[lc]].
template <typename V, typename U, typename G, typename SV>
__device__ __forceinline__ void light_tile(const LightStage<SV>& cur, int64_t t, int64_t nnz,
                                           const int32_t* __restrict__ light_cols,
                                           const U* u, G* out, int lane) {
  const unsigned FULL = 0xffffffffu;
  const int64_t a = t * kLightTile + (int64_t)lane * kLightItems;
  const bool active = a < nnz;
  const uint32_t m = cur.m, lc0 = cur.lc0;
  const int32_t* r = cur.r;
  const uint32_t cnt = __popc(lane == 0 ? (m & 0xfeu) : m);
  uint32_t incl = cnt;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const uint32_t y = __shfl_up_sync(FULL, incl, d);
    if (lane >= d) incl += y;
  }
  uint32_t q = lc0 + (incl - cnt) + (lane > 0 ? (m & 1u) : 0u);
  // columns this lane may write, loaded early
  const bool lead = lane == 0 && active && !(m & 1u);
  const uint32_t ql = q + __popc(m & 0xfeu);
  const int32_t j0 = lead ? __ldg(light_cols + lc0) : 0;
  const int32_t jl = (active && m != 0u) ? __ldg(light_cols + ql) : 0;
  V cont = V(0), tail = V(0);
  bool has_tail = false;
  if (active) {
    U uu[8];
#pragma unroll
    // gathers of u through L2 without allocating in L1 (no reuse to keep)
    for (int i = 0; i < 8; ++i) uu[i] = load_l2(u + r[i]);  // padding rows are 0, values 0
    // first run, last run and the whole columns between (see slab_pass)
    const uint32_t inner = m & 0xfeu;
    const int bf = inner ? __ffs(inner) - 1 : 8;
    V acc = V(0), first = V(0);
    uint32_t qi = q;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      if ((inner >> i) & 1u) {
        if (i == bf) {
          first = acc;
        } else {  // a whole column inside the lane
          out[__ldg(light_cols + qi)] = (G)acc;
        }
        acc = V(0);
        ++qi;
      }
      acc = fma((V)cur.val.get(i), (V)uu[i], acc);
    }
    if (inner) {
      if (m & 1u) {  // started at entry 0, ended inside
        out[__ldg(light_cols + q)] = (G)first;
      } else {
        cont = first;
      }
      tail = acc;
      has_tail = true;
    } else if (m & 1u) {
      tail = acc;
      has_tail = true;
    } else {
      cont = acc;
    }
  }
  const uint32_t stops = __ballot_sync(FULL, !active || m != 0u);
  if (stops == 0u) {
    const V sum = warp_sum(cont);  // the whole tile is inside column lc0
    if (lane == 0) atomicAdd(out + j0, (G)sum);
  } else {
    const V tsum = lane_suffix_sum(cont, stops, lane);
    const V t1s = __shfl_down_sync(FULL, tsum, 1);
    if (lead) atomicAdd(out + j0, (G)tsum);  // column from the previous tile
    if (has_tail) {
      const V sum = tail + (lane < 31 ? t1s : V(0));
      emit_pair<G>(out, (uint32_t)jl, (G)sum, lane < 31 && (stops >> (lane + 1)) != 0u);
    }
  }
}

template <typename V, typename U, typename G, typename SV>
__global__ void __launch_bounds__(kThreads, 3)
    k_propose_light_runs(const int32_t* __restrict__ row, const SV* __restrict__ val,
                         const uint8_t* __restrict__ lmask, const int32_t* __restrict__ tile_lc,
                         const int32_t* __restrict__ light_cols, const U* u, int64_t nnz, int64_t ntiles, G* out) {
  const int lane = threadIdx.x & 31;
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  pdl_trigger();
  constexpr bool kPrefetch = sizeof(V) == 4;  // FP64 stages are too large to double in registers
  LightStage<SV> nxt;
  if (kPrefetch) load_light_stage<SV>(row, val, lmask, tile_lc, warp, ntiles, nnz, lane, nxt);
  pdl_wait();
  for (int64_t t = warp; t < ntiles; t += nwarps) {  // warp-uniform
    LightStage<SV> cur;
    if (kPrefetch) {
      cur = nxt;
      load_light_stage<SV>(row, val, lmask, tile_lc, t + nwarps, ntiles, nnz, lane, nxt);  // next tile in flight
    } else {
      load_light_stage<SV>(row, val, lmask, tile_lc, t, ntiles, nnz, lane, cur);
    }
    light_tile<V, U, G, SV>(cur, t, nnz, light_cols, u, out, lane);
  }
}

// The light tiles as a shared pool: warps take kLightChunk tiles at a time
// from a global counter (reset by the last warp of k_propose_fused), the next
// tile's loads in flight while one is summed.
constexpr int kLightChunk = 4;

template <typename V, typename U, typename G, typename SV>
__device__ __forceinline__ void light_pool(const int32_t* __restrict__ row, const SV* __restrict__ val,
                                           const uint8_t* __restrict__ lmask, const int32_t* __restrict__ tile_lc,
                                           const int32_t* __restrict__ light_cols, const U* u, int64_t nnz,
                                           int64_t ntiles, G* out, unsigned int* counter) {
  const int lane = threadIdx.x & 31;
  auto grab = [&](int64_t& t, int64_t& t_end) {
    unsigned int b = 0;
    if (lane == 0) b = atomicAdd(counter, (unsigned int)kLightChunk);
    b = __shfl_sync(0xffffffffu, b, 0);
    t = (int64_t)b;
    t_end = t + kLightChunk < ntiles ? t + kLightChunk : ntiles;
  };
  int64_t t, t_end;
  grab(t, t_end);
  if (t >= ntiles) return;
  LightStage<SV> nxt;
  load_light_stage<SV>(row, val, lmask, tile_lc, t, ntiles, nnz, lane, nxt);
  for (;;) {  // warp-uniform
    const LightStage<SV> cur = nxt;
    const int64_t tc = t;
    if (++t >= t_end) grab(t, t_end);
    const bool more = t < ntiles;
    if (more) load_light_stage<SV>(row, val, lmask, tile_lc, t, ntiles, nnz, lane, nxt);  // next tile in flight
    light_tile<V, U, G, SV>(cur, tc, nnz, light_cols, u, out, lane);
    if (!more) break;
  }
}

// Both streaming passes in one persistent kernel, one CTA per SM: warps
// 0 .. SLAB_WARPS - 1 run the CTA's row-slab tiles (u slab in shared memory,
// synchronised on named barrier 1), the other warps take light tiles from
// the pool, and the slab warps join the pool when their tiles are done.  The
// slab pass waits on memory latency and the light pass on L1 gathers, so
// running them side by side on every SM overlaps the two.
template <typename V, typename U, typename G, int THREADS, int SLAB_WARPS, int DEPTH, int ITEMS, typename SV>
__global__ void __launch_bounds__(THREADS, 1)
    k_propose_fused(const uint16_t* __restrict__ s_row, const SV* __restrict__ s_val,
                    const uint8_t* __restrict__ pmask, const uint32_t* __restrict__ pair_col, SlabTiles T,
                    const int32_t* __restrict__ lrow, const SV* __restrict__ lval,
                    const uint8_t* __restrict__ lmask, const int32_t* __restrict__ tile_lc,
                    const int32_t* __restrict__ light_cols, int64_t lnnz,
                    int64_t lntiles, unsigned int* counter, const U* u, int64_t n, int32_t slab_rows, G* gacc,
                    int64_t second) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  U* s_u = reinterpret_cast<U*>(smem_raw);
  pdl_trigger();
  const int warp = threadIdx.x >> 5;
  if (warp < SLAB_WARPS)
    slab_pass<V, U, G, DEPTH, ITEMS, SV, 32 * SLAB_WARPS>(
        s_row, s_val, pmask, pair_col, T, T.cta_tile_begin[blockIdx.x], T.cta_tile_begin[blockIdx.x + 1], u, n,
        slab_rows, gacc, second, s_u, warp, SLAB_WARPS, threadIdx.x, 32 * SLAB_WARPS);
  else
    pdl_wait();
  light_pool<V, U, G, SV>(lrow, lval, lmask, tile_lc, light_cols, u, lnnz, lntiles, gacc, counter);
  // the last warp out resets the pool for the next launch: every warp has
  // taken its last tiles when it gets here (counter[1] counts the exits)
  if ((threadIdx.x & 31) == 0) {
    const unsigned int warps = gridDim.x * (THREADS / 32);
    __threadfence();  // this warp's takes from the pool are performed before its exit counts
    if (atomicAdd(counter + 1, 1u) == warps - 1) {
      counter[0] = 0u;
      counter[1] = 0u;
    }
  }
}

static SlabTiles tiles_of(const ProposePlan& P) {
  return SlabTiles{P.tile_pair, P.tile_slab, P.slab_tile_begin, P.cta_tile_begin, P.slab_off};
}

// the two streaming passes for one value storage SV (V compute type, U type
// of u, G accumulator)
constexpr int kFusedThreads = 1024;
// candidate splits of the fused kernel's 32 warps: warps that start on the
// row slabs (the rest start on the light pool); the plan's autotuner times
// each, and the two separate kernels, on the problem at hand
constexpr int kFusedSplits[] = {20, 24, 28, 31};
constexpr int kNumFusedSplits = 4;

template <typename V, typename U, typename G, typename SV, int SW>
static cudaError_t launch_fused(gencd_problem* p, const void* u_vec, size_t smem) {
  ProposePlan& P = p->plan;
  return launch_overlapped(k_propose_fused<V, U, G, kFusedThreads, SW, 1, kSlabItemsF32, SV>, P.grid, kFusedThreads, smem,
                           launch_on(p), P.s_row, (const SV*)P.s_val, P.pmask, P.pair_col, tiles_of(P),
                           P.light_row, (const SV*)P.light_val, P.lmask, P.light_tile_lc, P.light_cols,
                           P.light_nnz, P.light_ntiles, P.light_counter, (const U*)u_vec, p->n, P.slab_rows,
                           (G*)p->gnat, P.second);
}

// both passes in one kernel
template <typename V, typename U, typename G, typename SV>
static int launch_fused_passes(gencd_problem* p, const void* u_vec) {
  const size_t smem = (size_t)(p->plan.slab_rows + kSlabZeroSlot) * sizeof(U);
  cudaEvent_t e1 = nullptr;
  prof_begin(p, K_PROPOSE_FUSED, &e1);
  cudaError_t err;
  switch (p->plan.fused_split) {
    case 20: err = launch_fused<V, U, G, SV, 20>(p, u_vec, smem); break;
    case 24: err = launch_fused<V, U, G, SV, 24>(p, u_vec, smem); break;
    case 28: err = launch_fused<V, U, G, SV, 28>(p, u_vec, smem); break;
    default: err = launch_fused<V, U, G, SV, 31>(p, u_vec, smem); break;
  }
  prof_end(p, e1);
  GENCD_CUDA_TRY(err);
  return GENCD_OK;
}

template <typename V, typename U, typename G, typename SV, int THREADS, int DEPTH, int ITEMS>
static int launch_plan_passes(gencd_problem* p, const void* u_vec) {
  ProposePlan& P = p->plan;
  if constexpr (sizeof(V) == 4) {
    if (P.fused_split > 0) return launch_fused_passes<V, U, G, SV>(p, u_vec);
  }
  if (P.nlight > 0) {
    cudaEvent_t e = nullptr;
    prof_begin(p, K_PROPOSE_LIGHT, &e);
    const int grid = grid_for(P.light_ntiles * 32, kThreads, p->num_sms * 3);  // resident CTAs: persistent warps
    const cudaError_t err = launch_overlapped(
        k_propose_light_runs<V, U, G, SV>, grid, kThreads, 0, launch_on(p), P.light_row, (const SV*)P.light_val, P.lmask,
        P.light_tile_lc, P.light_cols, (const U*)u_vec, P.light_nnz, P.light_ntiles, (G*)p->gnat);
    prof_end(p, e);
    GENCD_CUDA_TRY(err);
  }
  if (P.nheavy > 0) {
    const size_t smem = (size_t)(P.slab_rows + kSlabZeroSlot) * sizeof(U);
    cudaEvent_t e1 = nullptr;
    prof_begin(p, K_PROPOSE_SLABS, &e1);
    const cudaError_t err = launch_overlapped(
        k_propose_slabs<V, U, G, THREADS, DEPTH, ITEMS, SV>, P.grid, THREADS, smem, launch_on(p), P.s_row,
        (const SV*)P.s_val, P.pmask, P.pair_col, tiles_of(P), (const U*)u_vec, p->n, P.slab_rows,
        (G*)p->gnat, P.second);
    prof_end(p, e1);
    GENCD_CUDA_TRY(err);
  }
  return GENCD_OK;
}

template <typename V, typename U, typename G, typename SV, int THREADS, int DEPTH, int ITEMS>
static int set_slab_smem(const ProposePlan& P) {
  // the limit belongs to the kernel, not to the problem: the largest slab's
  const int smem = (int)(kSlabBytes + kSlabZeroSlot * sizeof(U));
  GENCD_CUDA_TRY(cudaFuncSetAttribute(k_propose_slabs<V, U, G, THREADS, DEPTH, ITEMS, SV>,
                                      cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
  if constexpr (sizeof(V) == 4) {
    if (P.light_counter) {
      GENCD_CUDA_TRY(cudaFuncSetAttribute(k_propose_fused<V, U, G, kFusedThreads, 20, 1, kSlabItemsF32, SV>,
                                          cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
      GENCD_CUDA_TRY(cudaFuncSetAttribute(k_propose_fused<V, U, G, kFusedThreads, 24, 1, kSlabItemsF32, SV>,
                                          cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
      GENCD_CUDA_TRY(cudaFuncSetAttribute(k_propose_fused<V, U, G, kFusedThreads, 28, 1, kSlabItemsF32, SV>,
                                          cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
      GENCD_CUDA_TRY(cudaFuncSetAttribute(k_propose_fused<V, U, G, kFusedThreads, 31, 1, kSlabItemsF32, SV>,
                                          cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    }
  }
  return GENCD_OK;
}

#define GENCD_PLAN_F64 double, double, double, double, kSlabThreadsF64, kSlabDepthF64, kSlabItemsF64
#define GENCD_PLAN_F32(SV) float, float, float, SV, kSlabThreadsF32, kSlabDepthF32, kSlabItemsF32

int launch_propose_plan(gencd_problem* p, const void* u_vec) {
  if (p->precision == GENCD_F64) return launch_plan_passes<GENCD_PLAN_F64>(p, u_vec);
  if (p->vmode == kValBf16) return launch_plan_passes<GENCD_PLAN_F32(__nv_bfloat16)>(p, u_vec);
  if (p->vmode == kValNone) return launch_plan_passes<GENCD_PLAN_F32(NoVal)>(p, u_vec);
  return launch_plan_passes<GENCD_PLAN_F32(float)>(p, u_vec);
}

// ---------------------------------------------------------------------------
// building the plan (once per problem)

// What the choice of the heavy columns needs: out[0] columns that are not
// empty, out[1] entries of those shorter than hmin, out[2] and out[3] columns
// below and from `forms` entries
__global__ void __launch_bounds__(kThreads)
    k_plan_count(const int64_t* __restrict__ col_ptr, int64_t k, int64_t hmin, int64_t forms,
                 unsigned long long* __restrict__ out) {
  unsigned long long c[4] = {0, 0, 0, 0};
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < k; j += stride) {
    const int64_t len = col_ptr[j + 1] - col_ptr[j];
    if (len <= 0) continue;
    c[0] += 1;
    if (len < hmin) c[1] += (unsigned long long)len;
    c[len < forms ? 2 : 3] += 1;
  }
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    c[q] = warp_sum(c[q]);
    if ((threadIdx.x & 31) == 0 && c[q]) atomicAdd(out + q, c[q]);
  }
}

// Columns by kind, for the exclusive scans: hid and lid number the heavy and
// the light ones, loff offsets the light ones' entries.
__global__ void k_plan_classify(const int64_t* __restrict__ col_ptr, int64_t k, int64_t hmin,
                                uint32_t* __restrict__ hid, uint32_t* __restrict__ lid,
                                uint32_t* __restrict__ loff) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j <= k; j += stride) {
    const uint32_t len = j < k ? (uint32_t)(col_ptr[j + 1] - col_ptr[j]) : 0u;
    const bool heavy = len > 0 && (int64_t)len >= hmin;
    const bool light = len > 0 && !heavy;
    hid[j] = heavy;
    lid[j] = light;
    loff[j] = light ? len : 0u;
  }
}

__global__ void k_plan_columns(const int64_t* __restrict__ col_ptr, int64_t k, int64_t hmin,
                               const uint32_t* __restrict__ hid, const uint32_t* __restrict__ lid,
                               const uint32_t* __restrict__ loff, int32_t* __restrict__ heavy_cols,
                               int32_t* __restrict__ light_cols, int64_t* __restrict__ light_col_ptr) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j <= k; j += stride) {
    if (j == k) {
      light_col_ptr[lid[k]] = loff[k];
      continue;
    }
    const int64_t len = col_ptr[j + 1] - col_ptr[j];
    if (len <= 0) continue;
    if (len >= hmin) {
      heavy_cols[hid[j]] = (int32_t)j;
    } else {
      light_cols[lid[j]] = (int32_t)j;
      light_col_ptr[lid[j]] = loff[j];
    }
  }
}

template <typename T>
__global__ void k_plan_fill(T* __restrict__ a, int64_t m, T v) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < m; i += stride) a[i] = v;
}

// first entry of a column (rows r[0..len), ascending) at or beyond a row
__device__ __forceinline__ uint32_t rows_below(const int32_t* __restrict__ r, uint32_t len, int64_t row) {
  uint32_t lo = 0, hi = len;
  while (lo < hi) {
    const uint32_t mid = (lo + hi) >> 1;
    if ((int64_t)r[mid] < row)
      lo = mid + 1;
    else
      hi = mid;
  }
  return lo;
}

// The entries of heavy column h in slab r are one run of the column (its rows
// ascend).  Slab-major, i = r nheavy + h: seg[i] the run's first entry within
// the column, cnt[i] its length, pair[i] whether it is not empty (both for the
// exclusive scans; index count holds 0).
__global__ void k_plan_segments(const int64_t* __restrict__ col_ptr, const int32_t* __restrict__ row_idx,
                                const int32_t* __restrict__ heavy_cols, int64_t nheavy, int64_t count, int32_t R,
                                int32_t slab_rows, uint32_t* __restrict__ seg, uint32_t* __restrict__ cnt,
                                uint32_t* __restrict__ pair) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i <= count; i += stride) {
    uint32_t n_i = 0;
    if (i < count) {
      const int64_t r = i / nheavy;
      const int32_t j = heavy_cols[i - r * nheavy];
      const int64_t s = col_ptr[j];
      const uint32_t len = (uint32_t)(col_ptr[j + 1] - s);
      const uint32_t a = r == 0 ? 0u : rows_below(row_idx + s, len, r * slab_rows);
      const uint32_t b = r == R - 1 ? len : rows_below(row_idx + s, len, (r + 1) * slab_rows);
      seg[i] = a;
      n_i = b - a;
    }
    cnt[i] = n_i;
    pair[i] = n_i > 0 ? 1u : 0u;
  }
}

// entries before slab r (r = R: all of them), and the number of pairs
__global__ void k_plan_slab_begins(const uint32_t* __restrict__ pos, const uint32_t* __restrict__ pair, int64_t nheavy,
                                   int32_t R, int64_t* __restrict__ slab_begin) {
  for (int32_t r = threadIdx.x; r <= R; r += blockDim.x) slab_begin[r] = pos[(int64_t)r * nheavy];
  if (threadIdx.x == 0) slab_begin[R + 1] = pair[(int64_t)R * nheavy];
}

template <typename V>
__device__ __forceinline__ void plan_store(V* a, int64_t i, V v) {
  a[i] = v;
}
__device__ __forceinline__ void plan_store(__nv_bfloat16* a, int64_t i, float v) {
  a[i] = __float2bfloat16_rn(v);  // the values are bfloat16-exact
}
__device__ __forceinline__ void plan_store(NoVal*, int64_t, float) {}
template <typename SV>
__device__ __forceinline__ void plan_zero(SV* a, int64_t i) {
  a[i] = SV(0.0f);
}
__device__ __forceinline__ void plan_zero(NoVal*, int64_t) {}

// Every entry to its place: a heavy one into its slab's run (pad_off[r] is
// where the padded slab starts), a light one into the compact copy, in the
// plan's value storage; the start bits of pairs and light columns (bit p % 32
// of word p / 32 = bit p % 8 of byte p / 8), and each pair's first entry and
// column.
//
// Bound: memory.  Consecutive lanes take consecutive entries, so reads and, run
// by run, writes are coalesced; every entry finds its column within its tile
// (the tile map): 142 us on 2.0e7 FP32 non-zeros, 41 at the copy rate.  The
// entries' keys, order, rows, columns and values expanded (480 us: a warp walked
// a whole column), sorted by slab (117) and gathered (163), and the pairs (62),
// took 0.8 ms and 28 bytes of scratch a non-zero.
template <typename V, typename SV>
__global__ void __launch_bounds__(kThreads)
    k_plan_place(const int64_t* __restrict__ col_ptr, const int32_t* __restrict__ row_idx, const V* __restrict__ val,
                 const int32_t* __restrict__ tile_col, int64_t nnz, int64_t tile, int64_t hmin,
                 const uint32_t* __restrict__ hid, const uint32_t* __restrict__ loff, int64_t nheavy,
                 int32_t slab_rows, const uint32_t* __restrict__ seg, const uint32_t* __restrict__ pos,
                 const uint32_t* __restrict__ pair, const int64_t* __restrict__ slab_begin,
                 const int64_t* __restrict__ pad_off, uint16_t* __restrict__ s_row, SV* __restrict__ s_val,
                 uint32_t* __restrict__ pmask, uint32_t* __restrict__ pair_start, uint32_t* __restrict__ pair_col,
                 int32_t* __restrict__ lrow, SV* __restrict__ lval, uint32_t* __restrict__ lmask) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < nnz; p += stride) {
    const int64_t t = p / tile;
    int32_t lo = __ldg(tile_col + t), hi = __ldg(tile_col + t + 1);  // last c with col_ptr[c] <= p
    while (lo < hi) {
      const int32_t mid = (lo + hi + 1) >> 1;
      if (__ldg(col_ptr + mid) <= p)
        lo = mid;
      else
        hi = mid - 1;
    }
    const int64_t s = __ldg(col_ptr + lo), len = __ldg(col_ptr + lo + 1) - s;
    const int32_t row = row_idx[p];
    const uint32_t at = (uint32_t)(p - s);
    if (len >= hmin) {
      const int32_t r = row / slab_rows;
      const int64_t i = (int64_t)r * nheavy + __ldg(hid + lo);
      const uint32_t first = __ldg(seg + i);
      const int64_t d = __ldg(pad_off + r) - __ldg(slab_begin + r) + __ldg(pos + i) + (at - first);
      const int64_t d0 = d & ~(int64_t)(kSlabTile - 1);
      const uint32_t x = (uint32_t)(d - d0);
      s_row[d0 + slab_at<8>(x)] = (uint16_t)(row - r * slab_rows);
      plan_store(s_val, d0 + slab_at<vector_of<SV>()>(x), val[p]);
      if (at == first) {
        const uint32_t q = __ldg(pair + i);
        atomicOr(pmask + (d >> 5), 1u << (d & 31));
        pair_start[q] = (uint32_t)d;
        pair_col[q] = (uint32_t)lo;
      }
    } else {
      const int64_t d = (int64_t)__ldg(loff + lo) + at;
      lrow[d] = row;
      plan_store(lval, d, val[p]);
      if (at == 0) atomicOr(lmask + (d >> 5), 1u << (d & 31));
    }
  }
}

// the padding of every slab's last tile: the row past the slab, which reads a
// zero from shared memory, and value 0
template <typename SV>
__global__ void k_plan_pad(const int64_t* __restrict__ slab_begin, const int64_t* __restrict__ pad_off, int32_t R,
                           uint16_t pad_row, uint16_t* __restrict__ s_row, SV* __restrict__ s_val) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < (int64_t)R * kSlabTile; q += stride) {
    const int64_t r = q / kSlabTile, end = pad_off[r + 1];
    const uint32_t x = (uint32_t)(q - r * kSlabTile);  // place in the slab's last tile
    if (end == pad_off[r] || end - kSlabTile + x < pad_off[r] + (slab_begin[r + 1] - slab_begin[r])) continue;
    s_row[end - kSlabTile + slab_at<8>(x)] = pad_row;
    plan_zero(s_val, end - kSlabTile + slab_at<vector_of<SV>()>(x));
  }
}

__global__ void k_plan_tiles(const int32_t* __restrict__ slab_tile_begin, const int64_t* __restrict__ pad_off,
                             int32_t R, int64_t T, int64_t tile, const uint32_t* __restrict__ pair_start,
                             int64_t npairs, uint32_t* __restrict__ tile_pair, int32_t* __restrict__ tile_slab) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < T; t += stride) {
    int32_t lo = 0, hi = R - 1;  // slab: last r with slab_tile_begin[r] <= t
    while (lo < hi) {
      const int32_t mid = (lo + hi + 1) >> 1;
      if (slab_tile_begin[mid] <= t)
        lo = mid;
      else
        hi = mid - 1;
    }
    const int32_t r = lo;
    const int64_t s = pad_off[r] + (t - slab_tile_begin[r]) * tile;
    tile_slab[t] = r;
    int64_t a = 0, b = npairs - 1;  // pair of the tile's first entry: last q with pair_start[q] <= s
    while (a < b) {
      const int64_t mid = (a + b + 1) >> 1;
      if ((int64_t)pair_start[mid] <= s)
        a = mid;
      else
        b = mid - 1;
    }
    tile_pair[t] = (uint32_t)a;
  }
}

void free_propose_plan(gencd_problem* p) {
  for (void* b : p->plan.mem)
    if (b) dev_free(p, b);
  p->plan = ProposePlan();
}

// First tile of each of `grid` CTAs, from the slabs' first tiles tb[0..R].
// Equal runs of all tiles make some CTAs load two slabs of u, which takes as
// long as about kSlabSwitch entries; CTAs that keep to one slab have unequal
// runs.  The split whose longest CTA is shorter.
constexpr int64_t kSlabSwitch = 16384;

static std::vector<int32_t> split_tiles(const std::vector<int32_t>& tb, int grid, int64_t tile) {
  const int R = (int)tb.size() - 1;
  const int64_t T = tb[R];
  std::vector<int32_t> first(grid + 1);
  for (int b = 0; b <= grid; ++b) first[b] = (int32_t)(b * T / grid);
  if (R < 2 || R > grid || T == 0) return first;
  std::vector<int> ctas(R);  // proportional to the slabs' tiles, at least one each
  int left = grid;
  for (int r = 0; r < R; ++r) {
    ctas[r] = std::max<int>(1, (int)((int64_t)grid * (tb[r + 1] - tb[r]) / T));
    left -= ctas[r];
  }
  int64_t longest = 0;
  for (; left > 0; --left) {  // the rest to the slab with the longest runs
    int most = 0;
    for (int r = 1; r < R; ++r)
      if ((int64_t)(tb[r + 1] - tb[r]) * ctas[most] > (int64_t)(tb[most + 1] - tb[most]) * ctas[r]) most = r;
    ctas[most] += 1;
  }
  for (int r = 0; r < R; ++r) longest = std::max<int64_t>(longest, (tb[r + 1] - tb[r] + ctas[r] - 1) / ctas[r]);
  if (left < 0 || longest > (T + grid - 1) / grid + kSlabSwitch / tile) return first;
  int b = 0;
  for (int r = 0; r < R; ++r)
    for (int q = 0; q < ctas[r]; ++q)
      first[b++] = (int32_t)(tb[r] + (int64_t)q * (tb[r + 1] - tb[r]) / ctas[r]);
  return first;
}

// scratch that is freed when the build returns
struct Scratch {
  gencd_problem* p;
  std::vector<void*> bufs;
  explicit Scratch(gencd_problem* q) : p(q) {}
  int get(Arena& a) {
    void* base = nullptr;
    GENCD_TRY(dev_alloc_bytes(p, &base, a.bytes()));
    bufs.push_back(base);
    a.place(base);
    return GENCD_OK;
  }
  ~Scratch() {
    for (void* b : bufs) dev_free(p, b);
  }
};

template <typename V, typename SV>
static void launch_place(gencd_problem* p, const uint32_t* hid, const uint32_t* loff, const uint32_t* seg,
                         const uint32_t* pos, const uint32_t* pair, const int64_t* slab_begin, const int64_t* pad_off,
                         uint32_t* pair_start) {
  ProposePlan& P = p->plan;
  k_plan_place<V, SV><<<grid_for(p->nnz, kThreads, p->num_sms * 32), kThreads, 0, p->stream>>>(
      p->col_ptr, p->row_idx, (const V*)p->val, p->tile_col, p->nnz, 32LL * p->items, P.heavy_min, hid, loff, P.nheavy,
      P.slab_rows, seg, pos, pair, slab_begin, pad_off, P.s_row, (SV*)P.s_val, (uint32_t*)P.pmask, pair_start,
      P.pair_col, P.light_row, (SV*)P.light_val, (uint32_t*)P.lmask);
  if (P.nheavy > 0)
    k_plan_pad<SV><<<grid_for((int64_t)P.nslabs * kSlabTile, kThreads, p->num_sms * 8), kThreads, 0, p->stream>>>(
        slab_begin, pad_off, P.nslabs, (uint16_t)P.slab_rows, P.s_row, (SV*)P.s_val);
}

// Two allocations hold the plan and two the scratch: a cudaMalloc or cudaFree
// of this size takes longer than most of the kernels here (some forty of them
// took half of the 7 ms of a cold start on 2.0e7 non-zeros).
static int build_plan_impl(gencd_problem* p, Scratch& S) {
  ProposePlan& P = p->plan;
  const int64_t k = p->k, n = p->n;
  const bool f64 = p->precision == GENCD_F64;
  const size_t vsz = f64 ? 8 : p->vmode == kValBf16 ? 2 : p->vmode == kValNone ? 0 : 4;  // as the plan stores them
  const int g = p->num_sms * 8;
  cudaStream_t st = p->stream;
  // as few slabs as hold n rows, and all alike: a last slab with the few rows
  // left over has runs of one or two entries, whose sums and atomic adds made
  // its CTAs take 72 us where the others took 51 (4e7 non-zeros, n = 200,000:
  // 3,392 rows left).  Multiples of 8 rows keep the slabs' u 16-byte aligned.
  const int64_t most_rows = kSlabBytes / (f64 ? 8 : 4);
  P.nslabs = (int32_t)((n + most_rows - 1) / most_rows);
  P.slab_rows = (int32_t)(((n + P.nslabs - 1) / P.nslabs + 7) / 8 * 8);
  // Heavy columns.  One slab: every column.  Otherwise a column's run in a slab
  // costs about as much as gathering its entries from L2 (one L1 wavefront
  // each) once it averages half an entry per slab in FP32 arithmetic (uniform
  // columns, a pass over 9.0e7 and 1.8e7 entries as slabs / as light columns:
  // 1.4 a slab 255 / 343 us, 0.3 a slab 118 / 88) and two in FP64 (0.7 a slab 465
  // / 400).  The light pass is a kernel of its own, though: beside heavy columns,
  // what few entries would be left to it join the slabs (2e8 Zipf non-zeros: 4341
  // us for ten iterations from two a slab, 4106 from a half, 3772 with none left;
  // FP64 2e7 1137 / 1044), while the runs (R per column) are no more than the
  // non-zeros, which bounds the scratch of the build.  An iteration with three
  // columns of 20,000 beside uniform ones takes, in slabs / with the light pass,
  // 21.8 / 26.2 us (FP32, 1e5 columns of 3 over 7 slabs), 27.9 / 29.0 (1.9e5 of 8
  // over 21), 43.5 / 47.0 (FP64, 5e5 of 8 over 5); in FP64 it does not pay for
  // many entries at less than one a slab (9e4 columns of 40 over 41 slabs 45.0 /
  // 41.2; of 10 30.4 / 29.2, of 12 over 9 46.8 / 45.8).  Light columns alone
  // keep their pass, which is then the only kernel (FP32 19.5 / 19.4, 26.9 / 23.7;
  // FP64 44.1 / 41.7, 44.5 / 33.0 us).
  constexpr int64_t kFewLight = int64_t(1) << 22, kFewSparse = int64_t(1) << 20;
  // FP32 sums of many slabs go to two accumulators, odd slabs to the second: a
  // column's sums are added one after another, and two chains half as long keep
  // the error of short columns below that of the light pass, which adds in a
  // tree (columns of 30 over 21 slabs: 7.56e-8 of the norm with two, 8.74e-8 with
  // one, 7.52e-8 as light columns; Zipf columns in all 6.25e-8, 6.77e-8, 6.52e-8).
  // A run of one entry rounds its product once more than a lane's chain does:
  // uniform columns of 3 over 2 to 12 slabs 3.9e-8 to 4.2e-8 (light 3.7e-8), of 6
  // 4.6e-8 to 5.0e-8 (4.7e-8), of 12 and more as the light pass or less.
  P.second = !f64 && P.nslabs >= 8 ? k : 0;
  P.heavy_min = 1;
  P.forms = false;
  if (P.nslabs > 1) {
    P.heavy_min = f64 ? 2LL * P.nslabs : std::max<int64_t>(2, (P.nslabs + 1) / 2);
    unsigned long long* stats = nullptr;
    Arena count;
    count.add(&stats, 4);
    GENCD_TRY(S.get(count));
    GENCD_CUDA_TRY(cudaMemsetAsync(stats, 0, 4 * sizeof(*stats), st));
    k_plan_count<<<grid_for(k, kThreads, g), kThreads, 0, st>>>(p->col_ptr, k, P.heavy_min, 2LL * P.nslabs, stats);
    unsigned long long c[4];
    GENCD_CUDA_TRY(cudaMemcpyAsync(c, stats, sizeof(c), cudaMemcpyDeviceToHost, st));
    GENCD_CUDA_TRY(cudaStreamSynchronize(st));
    const int64_t columns = (int64_t)c[0], light = (int64_t)c[1], short_columns = (int64_t)c[2];  // FP64: the light ones
    if (light < p->nnz && light <= std::max(kFewLight, p->nnz / 10) &&
        columns * P.nslabs <= std::max(kFewLight, p->nnz) &&
        (!f64 || light <= kFewSparse || light >= short_columns * P.nslabs))
      P.heavy_min = 1;
    // the schedules of both passes stay selectable wherever columns lie on both
    // sides of two entries a slab, whether or not the rule leaves light ones
    P.forms = !f64 && c[2] > 0 && c[3] > 0;
  }

  // classify, number and offset the columns
  uint32_t *hid, *lid, *loff, *tmp;
  int32_t* heavy_cols;     // original column of heavy id h
  int64_t* light_col_ptr;  // of the light columns' copy
  Arena cols;
  cols.add(&heavy_cols, k);
  cols.add(&light_col_ptr, k + 1);
  cols.add(&hid, k + 1);
  cols.add(&lid, k + 1);
  cols.add(&loff, k + 1);
  cols.add(&tmp, scan_tmp_words(k + 1));
  GENCD_TRY(S.get(cols));
  k_plan_classify<<<grid_for(k + 1, kThreads, g), kThreads, 0, st>>>(p->col_ptr, k, P.heavy_min, hid, lid, loff);
  GENCD_TRY(exclusive_scan(p, hid, hid, k + 1, tmp));
  GENCD_TRY(exclusive_scan(p, lid, lid, k + 1, tmp));
  GENCD_TRY(exclusive_scan(p, loff, loff, k + 1, tmp));
  uint32_t tot[3];
  GENCD_CUDA_TRY(cudaMemcpyAsync(&tot[0], hid + k, 4, cudaMemcpyDeviceToHost, st));
  GENCD_CUDA_TRY(cudaMemcpyAsync(&tot[1], lid + k, 4, cudaMemcpyDeviceToHost, st));
  GENCD_CUDA_TRY(cudaMemcpyAsync(&tot[2], loff + k, 4, cudaMemcpyDeviceToHost, st));
  GENCD_CUDA_TRY(cudaStreamSynchronize(st));
  P.nheavy = tot[0];
  P.nlight = tot[1];
  P.light_nnz = tot[2];
  const int64_t E = p->nnz - P.light_nnz;  // heavy entries
  const int R = P.nslabs;
  const int64_t runs = (int64_t)R * P.nheavy;  // at most two per heavy entry (heavy_min), or p->nnz (or 2^22)

  // the plan's per-column arrays and the light columns' copy
  const int64_t lpad = P.nlight > 0 ? ((P.light_nnz + kPadNnz - 1) / kPadNnz) * kPadNnz + kPadNnz : 0;
  const int64_t lwords = (lpad + 31) / 32;  // start bits, one byte per 8 entries
  P.light_ntiles = (P.light_nnz + kLightTile - 1) / kLightTile;
  const bool fusable = P.forms;
  Arena light;
  light.add(&P.light_cols, P.nlight);
  light.add(&P.light_row, lpad);
  light.add((char**)&P.light_val, lpad * (int64_t)vsz);
  light.add(&P.light_tile_lc, P.light_ntiles + 1);
  light.add((uint32_t**)&P.lmask, lwords);
  if (fusable) light.add(&P.light_counter, 2);  // tiles taken, warps finished
  P.grid = p->num_sms;
  GENCD_TRY(dev_alloc_bytes(p, &P.mem[0], light.bytes()));
  light.place(P.mem[0]);
  k_plan_columns<<<grid_for(k + 1, kThreads, g), kThreads, 0, st>>>(p->col_ptr, k, P.heavy_min, hid, lid, loff,
                                                                     heavy_cols, P.light_cols, light_col_ptr);
  GENCD_CUDA_TRY(cudaGetLastError());
  if (P.nlight > 0) {
    if (p->vmode == kValNone) {  // padding has no value to zero it: it gathers u[n] = 0 instead
      k_plan_fill<int32_t><<<grid_for(lpad - P.light_nnz, kThreads, g), kThreads, 0, st>>>(
          P.light_row + P.light_nnz, lpad - P.light_nnz, (int32_t)n);
      GENCD_CUDA_TRY(cudaGetLastError());
    } else {
      GENCD_CUDA_TRY(cudaMemsetAsync(P.light_row + P.light_nnz, 0, sizeof(int32_t) * (lpad - P.light_nnz), st));
      GENCD_CUDA_TRY(cudaMemsetAsync((char*)P.light_val + vsz * P.light_nnz, 0, vsz * (lpad - P.light_nnz), st));
    }
    GENCD_CUDA_TRY(cudaMemsetAsync(P.lmask, 0, 4 * (size_t)lwords, st));
    GENCD_TRY(launch_tile_map_of(p, light_col_ptr, P.nlight, P.light_ntiles, P.light_tile_lc, kLightTile));
  }
  if (fusable) GENCD_CUDA_TRY(cudaMemsetAsync(P.light_counter, 0, 2 * sizeof(unsigned int), st));

  // the heavy columns' runs per slab, in slab order
  uint32_t *seg, *pos, *pair, *pair_start, *rtmp;
  int64_t *slab_begin, *pad_off;
  Arena heavy;
  heavy.add(&seg, runs);
  heavy.add(&pos, runs + 1);
  heavy.add(&pair, runs + 1);
  heavy.add(&pair_start, std::min(runs, E) + 1);  // a run that is not empty is a pair
  heavy.add(&rtmp, scan_tmp_words(runs + 1));
  heavy.add(&slab_begin, R + 2);
  heavy.add(&pad_off, R + 1);
  GENCD_TRY(S.get(heavy));
  std::vector<int64_t> hb(R + 2, 0), hp(R + 1, 0);
  if (P.nheavy > 0) {
    k_plan_segments<<<grid_for(runs + 1, kThreads, p->num_sms * 32), kThreads, 0, st>>>(
        p->col_ptr, p->row_idx, heavy_cols, P.nheavy, runs, R, P.slab_rows, seg, pos, pair);
    GENCD_TRY(exclusive_scan(p, pos, pos, runs + 1, rtmp));
    GENCD_TRY(exclusive_scan(p, pair, pair, runs + 1, rtmp));
    k_plan_slab_begins<<<1, kThreads, 0, st>>>(pos, pair, P.nheavy, R, slab_begin);
    GENCD_CUDA_TRY(cudaGetLastError());
    GENCD_CUDA_TRY(cudaMemcpyAsync(hb.data(), slab_begin, 8 * (R + 2), cudaMemcpyDeviceToHost, st));
    GENCD_CUDA_TRY(cudaStreamSynchronize(st));
  }
  P.npairs = hb[R + 1];
  for (int r = 0; r < R; ++r) hp[r + 1] = hp[r] + ((hb[r + 1] - hb[r] + kSlabPad - 1) / kSlabPad) * kSlabPad;
  P.entries = hp[R];
  const int64_t tile = 32LL * (f64 ? kSlabItemsF64 : kSlabItemsF32);
  if (P.entries >= (int64_t(1) << 32)) return fail_plan("heavy entries exceed 2^32");

  if (P.nheavy > 0) {
    // tiles inside each slab, and contiguous runs of tiles per CTA
    const int64_t mask_words = (P.entries + 31) / 32;  // start bits: one byte per 8 entries
    std::vector<uint32_t> off(R + 1);
    for (int r = 0; r <= R; ++r) off[r] = (uint32_t)hp[r];
    Arena slabs;
    slabs.add(&P.s_row, P.entries);
    slabs.add((char**)&P.s_val, P.entries * (int64_t)vsz);
    slabs.add((uint32_t**)&P.pmask, mask_words);
    slabs.add(&P.pair_col, P.npairs);
    slabs.add(&P.slab_off, R + 1);
    P.ntiles = P.entries / tile;
    slabs.add(&P.tile_pair, P.ntiles);
    slabs.add(&P.tile_slab, P.ntiles);
    slabs.add(&P.slab_tile_begin, R + 1);
    slabs.add(&P.cta_tile_begin, P.grid + 1);
    GENCD_TRY(dev_alloc_bytes(p, &P.mem[1], slabs.bytes()));
    slabs.place(P.mem[1]);
    GENCD_CUDA_TRY(cudaMemcpyAsync(pad_off, hp.data(), 8 * (R + 1), cudaMemcpyHostToDevice, st));
    GENCD_CUDA_TRY(cudaMemcpyAsync(P.slab_off, off.data(), 4 * (R + 1), cudaMemcpyHostToDevice, st));
    GENCD_CUDA_TRY(cudaMemsetAsync(P.pmask, 0, 4 * (size_t)mask_words, st));
    std::vector<int32_t> tb(R + 1);
    for (int r = 0; r <= R; ++r) tb[r] = (int32_t)(hp[r] / tile);
    const std::vector<int32_t> ctb = split_tiles(tb, P.grid, tile);
    GENCD_CUDA_TRY(cudaMemcpyAsync(P.slab_tile_begin, tb.data(), 4 * (R + 1), cudaMemcpyHostToDevice, st));
    GENCD_CUDA_TRY(cudaMemcpyAsync(P.cta_tile_begin, ctb.data(), 4 * (P.grid + 1), cudaMemcpyHostToDevice, st));
    GENCD_CUDA_TRY(cudaStreamSynchronize(st));  // the host arrays go here
  }
  if (p->nnz > 0) {
    if (f64)
      launch_place<double, double>(p, hid, loff, seg, pos, pair, slab_begin, pad_off, pair_start);
    else if (p->vmode == kValBf16)
      launch_place<float, __nv_bfloat16>(p, hid, loff, seg, pos, pair, slab_begin, pad_off, pair_start);
    else if (p->vmode == kValNone)
      launch_place<float, NoVal>(p, hid, loff, seg, pos, pair, slab_begin, pad_off, pair_start);
    else
      launch_place<float, float>(p, hid, loff, seg, pos, pair, slab_begin, pad_off, pair_start);
    GENCD_CUDA_TRY(cudaGetLastError());
  }
  P.fused_split = 0;
  if (P.nheavy > 0) {
    k_plan_tiles<<<grid_for(P.ntiles, kThreads, g), kThreads, 0, st>>>(P.slab_tile_begin, pad_off, R, P.ntiles, tile,
                                                                      pair_start, P.npairs, P.tile_pair, P.tile_slab);
    GENCD_CUDA_TRY(cudaGetLastError());
    // both passes may run in one kernel when there are light and heavy columns
    // (FP32 arithmetic: FP64 stages do not fit the fused kernel's registers);
    // the autotuner below decides
    if (f64)
      GENCD_TRY(set_slab_smem<GENCD_PLAN_F64>(P));
    else if (p->vmode == kValBf16)
      GENCD_TRY(set_slab_smem<GENCD_PLAN_F32(__nv_bfloat16)>(P));
    else if (p->vmode == kValNone)
      GENCD_TRY(set_slab_smem<GENCD_PLAN_F32(NoVal)>(P));
    else
      GENCD_TRY(set_slab_smem<GENCD_PLAN_F32(float)>(P));
  }
  GENCD_CUDA_TRY(cudaStreamSynchronize(st));  // scratch and the host arrays go when this returns
  p->prof.launches[K_SETUP] += 7;
  return GENCD_OK;
}

int build_propose_plan(gencd_problem* p) {
  free_propose_plan(p);
  int rc;
  {
    Scratch S(p);
    rc = build_plan_impl(p, S);
    if (rc != GENCD_OK) cudaStreamSynchronize(p->stream);
  }
  if (rc != GENCD_OK) {
    free_propose_plan(p);
    return rc;
  }
  p->plan.built = true;
  return tune_propose_plan(p);
}

// Autotuner of the streaming propose: times the separate light and slab
// kernels and every split of the fused kernel on this problem (CUDA events, u
// as it stands: one launch each, then two more of those within kTuneClose of
// the fastest) and keeps the fastest.  All candidates compute the same sums;
// the scratch they leave is cleared.
constexpr float kTuneClose = 1.15f;

int tune_propose_plan(gencd_problem* p) {
  constexpr int C = kNumFusedSplits + 1;
  ProposePlan& P = p->plan;
  for (double& ms : P.tuned_ms) ms = -1.0;
  P.fused_split = 0;
  if (!P.built || !P.light_counter || P.nlight == 0) return GENCD_OK;
  cudaEvent_t ev[2 * C] = {};
  int rc = GENCD_OK;
  for (cudaEvent_t& e : ev)
    if (rc == GENCD_OK && cudaEventCreate(&e) != cudaSuccess) rc = fail_plan("cudaEventCreate failed");
  const bool prof = p->prof.enabled;
  p->prof.enabled = false;
  const int kept = P.fused_split;
  auto form = [](int c) { return c == 0 ? 0 : kFusedSplits[c - 1]; };
  bool runs[C];
  int reps[C] = {};
  float total[C] = {};
  for (bool& r : runs) r = true;
  // each form once untimed (the first launch loads it), then the timed launches
  for (int pass = 0; pass < 3 && rc == GENCD_OK; ++pass) {
    const int n_launch = pass == 2 ? 2 : 1;
    for (int c = 0; c < C && rc == GENCD_OK; ++c) {
      if (!runs[c]) continue;
      P.fused_split = form(c);
      if (pass > 0) cudaEventRecord(ev[2 * c], p->stream);
      for (int r = 0; r < n_launch && rc == GENCD_OK; ++r) rc = launch_propose_plan(p, p->u);
      if (pass > 0) cudaEventRecord(ev[2 * c + 1], p->stream);
    }
    if (rc != GENCD_OK || pass == 0) continue;
    if (cudaStreamSynchronize(p->stream) != cudaSuccess) {
      rc = fail_plan("autotuning the streaming propose failed");
      break;
    }
    float best = 0.f;
    for (int c = 0; c < C; ++c) {
      if (!runs[c]) continue;
      float ms = 0.f;
      cudaEventElapsedTime(&ms, ev[2 * c], ev[2 * c + 1]);
      total[c] += ms;
      reps[c] += n_launch;
      P.tuned_ms[c] = total[c] / reps[c];
      if (c == 0 || (float)P.tuned_ms[c] < best) best = (float)P.tuned_ms[c];
    }
    for (int c = 0; c < C; ++c) runs[c] = (float)P.tuned_ms[c] <= kTuneClose * best;
  }
  int best = 0;
  for (int c = 1; c < C; ++c)
    if (P.tuned_ms[c] < P.tuned_ms[best]) best = c;
  p->prof.enabled = prof;
  P.fused_split = rc == GENCD_OK ? form(best) : kept;
  for (cudaEvent_t e : ev)
    if (e) cudaEventDestroy(e);
  if (rc != GENCD_OK) return rc;
  // the candidates' sums are scratch: the hot path expects them zero
  const size_t gsz = p->precision == GENCD_F64 ? sizeof(double) : sizeof(float);
  GENCD_CUDA_TRY(cudaMemsetAsync(p->gnat, 0, gsz * (size_t)(p->k + P.second), p->stream));
  return GENCD_OK;
}

}  // namespace gencd
