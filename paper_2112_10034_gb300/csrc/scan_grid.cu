// cox_scan: block-scope and grid-scope inclusive / exclusive scans.
//
// BLOCK scope follows the SDK's shfl_scan_test (Table 1 of the paper): each
// warp scans its 32 elements with shfl_up (Hillis-Steele), warp totals go to
// shared memory, warp 0 scans them, and every element takes its warp's
// prefix (the uniform_add step).
//
// GRID scope chains tiles.  16-byte aligned arrays take the row-tile kernels
// (k_scan_grid_rows and k_scan_grid_short, below); in any other layout tiles
// are chained by a decoupled look-back: a CTA takes a tile (16384 elements;
// 8192 for compensated sums, whose pairs need twice the shared memory) from an
// atomic ticket, receives it by plain loads (or one TMA bulk copy),
// and every warp scans its rows of 32 elements with shfl_up, carrying row
// totals across its rows (eight rows at a time for instruction-level
// parallelism).  Lane 0 of warp 0 scans the eight warp totals, the tile
// publishes its aggregate, walks back for its prefix, and every element
// takes prefix op warp-prefix op its value.  Each tile keeps its aggregate
// and its inclusive prefix in separate slots, each written before its flag
// (release store) and read after it (acquire load), so a reader never sees a
// value from the wrong stage.
#include <type_traits>

#include "cox_common.cuh"
#include "tile_pipe.cuh"

namespace cox {

constexpr size_t kScanWsHeader = 256;
constexpr int kScanLookV = 4;

__device__ __forceinline__ uint32_t ld_acquire_u32(const uint32_t* p) {
  uint32_t v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_release_u32(uint32_t* p, uint32_t v) {
  asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

template <class R>
__device__ __forceinline__ uint64_t pack(typename R::V v) {
  if constexpr (R::kComp) return (uint64_t)__float_as_uint(v.s) | ((uint64_t)__float_as_uint(v.e) << 32);
  else return (uint64_t)to_bits(v);
}
template <class R>
__device__ __forceinline__ typename R::V unpack(uint64_t u) {
  using T = typename R::T;
  if constexpr (R::kComp) return Pair{__uint_as_float((uint32_t)u), __uint_as_float((uint32_t)(u >> 32))};
  else return from_bits<T>((uint32_t)u);
}
template <class R>
__device__ __forceinline__ typename R::V warp_fold(typename R::V v) {
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) v = R::op(v, R::shfl_xor(v, off));
  return v;
}

// Look-back for generic scan values.  flags[t]: 0 nothing, 1 aggregate in
// agg[t], 2 inclusive prefix in inc[t].  Returns the tile's exclusive prefix.
template <class R>
__device__ typename R::V look_back_op(uint32_t* flags, uint64_t* agg, uint64_t* inc, int64_t tile,
                                      typename R::V total, uint32_t limit, unsigned* status, bool& gave_up) {
  using V = typename R::V;
  const int lane = lane_id();
  gave_up = false;
  if (tile == 0) {
    if (lane == 0) {
      st_relaxed_u64(inc, pack<R>(total));
      st_release_u32(flags, 2u);
    }
    return R::ident();
  }
  if (lane == 0) {
    st_relaxed_u64(agg + tile, pack<R>(total));
    st_release_u32(flags + tile, 1u);
  }
  V prefix = R::ident();
  uint32_t polls = 0;
  bool timed_out = false;
  for (int64_t w0 = tile - 1;; w0 -= 32 * kScanLookV) {
    uint32_t f[kScanLookV];
    uint64_t val[kScanLookV];
#pragma unroll
    for (int v = 0; v < kScanLookV; ++v) {
      const int64_t i = w0 - (lane * kScanLookV + v);
      f[v] = i >= 0 ? ld_acquire_u32(flags + i) : 2u;  // before tile 0: the identity
      val[v] = 0;
    }
    int lp;
    unsigned pm;
    for (;;) {
      lp = kScanLookV;
#pragma unroll
      for (int v = kScanLookV - 1; v >= 0; --v)
        if (f[v] == 2u) lp = v;
      pm = __ballot_sync(kFull, lp < kScanLookV);
      const int fl = pm ? __ffs(pm) - 1 : 32;
      bool missing = false;
#pragma unroll
      for (int v = 0; v < kScanLookV; ++v)
        if ((lane < fl || (lane == fl && v <= lp)) && f[v] == 0u) missing = true;
      if (!__any_sync(kFull, missing)) break;
      if (++polls > limit) {
        timed_out = true;
        break;
      }
      if (polls > 64) __nanosleep(100);
#pragma unroll
      for (int v = 0; v < kScanLookV; ++v) {
        const int64_t i = w0 - (lane * kScanLookV + v);
        if (f[v] == 0u && i >= 0) f[v] = ld_acquire_u32(flags + i);
      }
    }
    if (timed_out) break;
    const int fl = pm ? __ffs(pm) - 1 : 32;
    V part = R::ident();
#pragma unroll
    for (int v = kScanLookV - 1; v >= 0; --v) {  // older tiles first
      const int64_t i = w0 - (lane * kScanLookV + v);
      if (lane < fl || (lane == fl && v <= lp)) {
        const V x = i < 0 ? R::ident() : unpack<R>(ld_relaxed_u64((f[v] == 2u ? inc : agg) + i));
        part = R::op(x, part);
      }
    }
    prefix = R::op(warp_fold<R>(part), prefix);
    if (pm) break;
  }
  if (__any_sync(kFull, timed_out)) {
    gave_up = true;
    if (lane == 0) {
      atomicOr(status, (unsigned)kDevTimeout);
      st_relaxed_u64(inc + tile, pack<R>(total));  // release successors
      st_release_u32(flags + tile, 2u);
    }
    return R::ident();
  }
  if (lane == 0) {
    st_relaxed_u64(inc + tile, pack<R>(R::op(prefix, total)));
    st_release_u32(flags + tile, 2u);
  }
  return prefix;
}

// Published tile aggregates of the row-tile kernels, zero until written.  A
// 32-bit value is one 64-bit word, (1 << 32) | bits; a compensated pair two,
// one per 32-bit half, each with its own flag, so that every word read is
// whole whatever order the halves arrive in.  PK: a pair in one word -- a flag
// in bit 62, the error word rounded to 21 mantissa bits (about 2^-46 of the
// sum) above the sum word -- for workspaces smaller than cox_scan_workspace().
template <class R, bool PK>
__host__ __device__ constexpr int agg_words() {
  return R::kComp && !PK ? 2 : 1;
}
template <class R, bool PK>
__device__ __forceinline__ void agg_store(uint64_t* agg, int64_t tile, typename R::V v) {
  if constexpr (R::kComp && PK)
    // (a carry of the rounding into the exponent is the next binade's value)
    st_relaxed_u64(agg + tile, (1ull << 62) | ((((uint64_t)__float_as_uint(v.e) + 2u) >> 2 & 0x3FFFFFFFull) << 32) |
                                   __float_as_uint(v.s));
  else if constexpr (R::kComp)
    asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(agg + 2 * tile),
                 "l"((1ull << 32) | __float_as_uint(v.s)), "l"((1ull << 32) | __float_as_uint(v.e))
                 : "memory");
  else
    st_relaxed_u64(agg + tile, (1ull << 32) | to_bits(v));
}
// The aggregate as two flagged halves (a 32-bit value twice), zero flags while
// it is not there.
template <class R, bool PK>
__device__ __forceinline__ void agg_load(const uint64_t* agg, int64_t tile, uint64_t (&w)[2]) {
  if constexpr (R::kComp && PK) {
    const uint64_t q = ld_relaxed_u64(agg + tile), flag = (q >> 62) << 32;
    w[0] = flag | (uint32_t)q;
    w[1] = flag | (uint32_t)((uint32_t)(q >> 32) << 2);
  } else if constexpr (R::kComp) {
    asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(w[0]), "=l"(w[1]) : "l"(agg + 2 * tile) : "memory");
  } else {
    w[0] = w[1] = ld_relaxed_u64(agg + tile);
  }
}
template <class R>
__device__ __forceinline__ typename R::V agg_value(const uint64_t (&w)[2]) {
  if constexpr (R::kComp) return Pair{__uint_as_float((uint32_t)w[0]), __uint_as_float((uint32_t)w[1])};
  else return from_bits<typename R::T>((uint32_t)w[0]);
}

// Look-back of the short form's 32-bit sums (wrapping adds, so that a group's
// sum can be taken by atomics in any order): desc[t] = (state << 32) | value,
// state 0 nothing, 1 aggregate, 2 inclusive prefix.  Tiles form groups of 32;
// a tile adds (1 << 48) | value to its group's accumulator gacc[g] after
// publishing its aggregate, and the add that completes the group publishes the
// group aggregate in gdesc[g]; the last tile of a group also puts its
// inclusive prefix there (atomicMax: a state-2 word is larger than any state-1
// word).  The look-back reads the tile's own group first, then whole groups,
// 32 per window (1024 tiles): a few lines, where reading every earlier
// aggregate has all CTAs poll all lines while they are being written.  Called
// by a whole warp; a wait that runs out publishes a zero prefix.
__device__ unsigned look_back_sum2(uint64_t* desc, uint64_t* gdesc, uint64_t* gacc, int64_t tile, int64_t ntiles,
                                   unsigned total, uint32_t limit, unsigned* status, bool& gave_up) {
  const int lane = lane_id();
  gave_up = false;
  const int64_t g = tile >> 5;
  const int pos = (int)(tile & 31);
  if (lane == 0) {
    st_relaxed_u64(desc + tile, ((tile == 0 ? 2ull : 1ull) << 32) | total);
    const int64_t gsize = min((int64_t)32, ntiles - (g << 5));
    const unsigned long long old = atomicAdd(reinterpret_cast<unsigned long long*>(gacc + g), (1ull << 48) | total);
    if ((int64_t)(old >> 48) + 1 == gsize)
      atomicMax(reinterpret_cast<unsigned long long*>(gdesc + g), (1ull << 32) | (uint32_t)(old + total));
  }
  unsigned prefix = 0;
  uint32_t polls = 0;
  bool timed_out = false;
  bool done = tile == 0;
  if (!done && pos > 0) {  // own group: lane l holds position l < pos
    const int64_t g0 = g << 5;
    uint64_t d = lane < pos ? ld_relaxed_u64(desc + g0 + lane) : (1ull << 32);
    unsigned pm;
    int fl;
    for (;;) {
      pm = __ballot_sync(kFull, lane < pos && (d >> 32) == 2u);
      fl = pm ? 31 - __clz(pm) : -1;
      const bool missing = lane < pos && lane > fl && (d >> 32) == 0u;
      if (!__any_sync(kFull, missing)) break;
      if (++polls > limit) {
        timed_out = true;
        break;
      }
      if (polls > 64) __nanosleep(64);
      if (missing) d = ld_relaxed_u64(desc + g0 + lane);
    }
    if (!__any_sync(kFull, timed_out)) {
      unsigned v = (lane < pos && lane >= fl) ? (unsigned)d : 0u;
      prefix = __reduce_add_sync(kFull, v);
      done = fl >= 0;
    }
  }
  if (!done && !__any_sync(kFull, timed_out)) {  // whole groups: lane l holds group gw - l
    for (int64_t gw = g - 1;; gw -= 32) {
      const int64_t gi = gw - lane;
      uint64_t d = gi >= 0 ? ld_relaxed_u64(gdesc + gi) : (2ull << 32);  // before group 0: 0
      unsigned pm;
      for (;;) {
        pm = __ballot_sync(kFull, (d >> 32) == 2u);
        const int fl = pm ? __ffs(pm) - 1 : 32;
        const bool missing = lane <= fl && (d >> 32) == 0u;
        if (!__any_sync(kFull, missing)) break;
        if (++polls > limit) {
          timed_out = true;
          break;
        }
        if (polls > 64) __nanosleep(64);
        if (missing && gi >= 0) d = ld_relaxed_u64(gdesc + gi);
      }
      if (__any_sync(kFull, timed_out)) break;
      const int fl = pm ? __ffs(pm) - 1 : 32;
      prefix += __reduce_add_sync(kFull, lane <= fl ? (unsigned)d : 0u);
      if (pm) break;
    }
  }
  if (__any_sync(kFull, timed_out)) {
    gave_up = true;
    if (lane == 0) {
      atomicOr(status, (unsigned)kDevTimeout);
      st_relaxed_u64(desc + tile, (2ull << 32) | total);
      if (pos == 31) atomicMax(reinterpret_cast<unsigned long long*>(gdesc + g), (2ull << 32) | total);
    }
    return 0u;
  }
  if (lane == 0) {
    const uint64_t inc = (2ull << 32) | (uint32_t)(prefix + total);
    if (tile != 0) st_relaxed_u64(desc + tile, inc);
    if (pos == 31) atomicMax(reinterpret_cast<unsigned long long*>(gdesc + g), inc);
  }
  return prefix;
}

// Shape of the row-tile kernel, one CTA per SM.  32-bit values are bound by
// memory: 9 tiles of 24 KB (192 rows) run 2^28 int32 in 312-321 us, 6 of 32 KB
// 331, 12 of 16 KB 430 (a prefix per tile becomes the limit).  Compensated
// sums are bound by the prefix walk, whose combines are eight adds: 6 tiles of
// 32 KB, 2^27 in 185 us, 8 of 24 KB 217.  Two or three loads in flight keep
// memory busy; without a limit they wait for each other, in an order that is
// not the tiles' (2^28 int32, 32 KB tiles: 331 us with two, 359 with six).
template <class R>
struct GridCfg {
  static constexpr int kRows = R::kComp ? 256 : 192;  // rows per tile and TMA box
  static constexpr uint32_t kTileBytes = kRows * 128;
  static constexpr int kNB = R::kComp ? 6 : 9;      // tiles in shared memory
  static constexpr int kNW = kRows / 32;            // worker warps
  static constexpr int kWin = 8;                    // 32-tile rows per poll of the walk
  static constexpr int kFlight = R::kComp ? 2 : 3;  // loads in flight
  static constexpr int kThreads = (kNW + 3) * 32;
};

// A walk over the published aggregates in tile order (a whole warp): advances
// from `cur` to `tile`, folding what it passes into `run`.  False if the
// words did not appear within `limit` polls or `abort` was raised.
template <class R, bool PK>
__device__ bool follow(const uint64_t* agg, int64_t tile, int64_t& cur, typename R::V& run, uint32_t limit,
                       volatile int* abort) {
  using V = typename R::V;
  constexpr int kWin = GridCfg<R>::kWin;  // 32-tile rows per poll
  const int lane = lane_id();
  uint32_t polls = 0;
  while (cur < tile) {
    uint64_t w[kWin][2];
#pragma unroll
    for (int v = 0; v < kWin; ++v) {
      const int64_t t = cur + v * 32 + lane;
      w[v][0] = w[v][1] = 0;
      if (t < tile) agg_load<R, PK>(agg, t, w[v]);
    }
    V part = R::ident();
    int64_t step = 0;
#pragma unroll
    for (int v = 0; v < kWin; ++v) {
      if (step != v * 32) break;  // (a gap in an earlier row)
      const unsigned there = __ballot_sync(kFull, (w[v][0] >> 32) != 0 && (w[v][1] >> 32) != 0);
      const int n = there == kFull ? 32 : __ffs(~there) - 1;
      if (lane < n) part = R::op(part, agg_value<R>(w[v]));
      step += n;
    }
    if (step) {
      run = R::op(run, warp_fold<R>(part));
      cur += step;
      polls = 0;
      continue;
    }
    if (++polls > limit || __any_sync(kFull, *abort)) return false;
    __nanosleep(polls > 64 ? 200 : 20);
  }
  return true;
}

template <class R>
__host__ __device__ constexpr int grid_scan_tile() {
  return R::kComp ? 8192 : 16384;
}

template <class R>
__global__ void __launch_bounds__(256) k_scan_grid(const uint32_t* __restrict__ in, uint32_t* __restrict__ out,
                                                   int64_t n, unsigned* ticket, uint32_t* flags, uint64_t* agg,
                                                   uint64_t* inc, int64_t ntiles, int excl, uint32_t limit,
                                                   unsigned* status, int vec) {
  using T = typename R::T;
  using V = typename R::V;
  constexpr int TILE = grid_scan_tile<R>();
  constexpr int NW = 8;
  constexpr int RPW = TILE / 32 / NW;  // rows per warp
  extern __shared__ __align__(16) uint32_t smem[];
  uint32_t* bs = smem;                                        // values (or sum words)
  float* be = reinterpret_cast<float*>(smem + TILE);          // error words (compensated)
  uint64_t* bar = reinterpret_cast<uint64_t*>(smem + TILE * (R::kComp ? 2 : 1));
  __shared__ V s_wtot[NW], s_cp[NW];
  __shared__ int64_t s_tile;
  __shared__ int s_bad;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (tid == 0) {
    s_tile = atomicAdd(ticket, 1u);
    mbar_init(bar, 1);
    mbar_init_fence();
  }
  __syncthreads();
  const int64_t tile = s_tile;
  if (tile >= ntiles) return;
  const int64_t base = tile * TILE;
  const int valid = (int)min((int64_t)TILE, n - base);
  if (vec && valid == TILE) {
    if (tid == 0) {
      mbar_arrive_expect_tx(bar, (uint32_t)(TILE * 4));
      tma_load_1d(bs, in + base, (uint32_t)(TILE * 4), bar);
    }
    const bool ok = mbar_wait_bounded(bar, 0u, limit);
    if (__syncthreads_or(!ok)) {
      if (tid == 0) {
        atomicOr(status, (unsigned)kDevTimeout);
        mbar_drain(bar, 0u);
        st_relaxed_u64(inc + tile, pack<R>(R::ident()));
        st_release_u32(flags + tile, 2u);
      }
      return;
    }
  } else {
    const uint32_t pad = to_bits(R::pad());
    for (int i = tid; i < TILE; i += blockDim.x) bs[i] = i < valid ? in[base + i] : pad;
    __syncthreads();
  }
  // rows of warp w: w*RPW .. w*RPW + RPW - 1, eight at a time
  V carry = R::ident();
#pragma unroll 1
  for (int g = 0; g < RPW / 8; ++g) {
    V v[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = R::load(from_bits<T>(bs[(warp * RPW + g * 8 + i) * 32 + lane]));
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const V u = R::shfl_up_fresh(v[i], 1, 32);
      if (lane >= 1) v[i] = R::op_fresh(u, v[i]);
    }
#pragma unroll
    for (int d = 2; d < 32; d <<= 1) {
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const V u = R::shfl_up(v[i], d, 32);
        if (lane >= d) v[i] = R::op(u, v[i]);
      }
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) {  // carry the running total into each row
      const V tot = R::shfl_idx(v[i], 31, 32);
      v[i] = R::op(carry, v[i]);
      carry = R::op(carry, tot);
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int idx = (warp * RPW + g * 8 + i) * 32 + lane;
      if constexpr (R::kComp) {
        bs[idx] = __float_as_uint(v[i].s);
        be[idx] = v[i].e;
      } else {
        bs[idx] = to_bits(v[i]);
      }
    }
  }
  if (lane == 0) s_wtot[warp] = carry;
  __syncthreads();
  if (warp == 0) {
    V total = R::ident();
    if (lane == 0) {
#pragma unroll
      for (int k = 0; k < NW; ++k) {
        s_cp[k] = total;  // warp-exclusive prefix for now
        total = R::op(total, s_wtot[k]);
      }
    }
    total = R::shfl_idx(total, 0, 32);
    bool gave_up;
    const V prefix = look_back_op<R>(flags, agg, inc, tile, total, limit, status, gave_up);
    if (lane == 0) {
#pragma unroll
      for (int k = 0; k < NW; ++k) s_cp[k] = R::op(prefix, s_cp[k]);
      s_bad = gave_up;
    }
  }
  __syncthreads();
  if (s_bad) return;
  const V cp = s_cp[warp];
  auto value = [&](int idx) -> V {
    if constexpr (R::kComp) return Pair{__uint_as_float(bs[idx]), be[idx]};
    else return from_bits<T>(bs[idx]);
  };
  const int first = warp * RPW * 32;
#pragma unroll 4
  for (int rr = 0; rr < RPW; ++rr) {
    const int idx = (warp * RPW + rr) * 32 + lane;
    const int64_t gi = base + idx;
    T y;
    if (!excl) y = R::out(R::op(cp, value(idx)));
    else y = idx == first ? R::out(cp) : R::out(R::op(cp, value(idx - 1)));
    if (gi < n) out[gi] = to_bits(y);
  }
}

// GRID scope over aligned arrays of at least one full row, through tile_pipe:
// a tile of 192 rows of 32 elements (compensated pairs and short arrays: 256)
// arrives by one 2D TMA box with 128-byte swizzle; lane t of worker w owns row
// 32 w + t of the tile.  fold: each lane folds its row, a shuffle scan over the
// warp's rows gives every row's exclusive prefix in the warp; publish: the scan
// of the warp totals (one per 32 rows), the tile's aggregate; prefix: the walk
// over the earlier tiles' aggregates;
// finish: re-reads the row, carrying prefix op value into each element (in
// place), before one TMA store.  Sums are folded left to right within a row,
// so fp32 results differ from the shuffle form in their last bits
// (tolerance-checked).  The partial last row (n % 32 elements) is read and
// written by its lane from global memory.
// a op x for one element x: for a compensated pair the element's error word
// is zero, so the error words need one add (a.e + t), not two.
template <class R>
__device__ __forceinline__ typename R::V op_elem(typename R::V a, typename R::T x) {
  if constexpr (R::kComp) {
    Pair r;
    float t;
    two_sum(a.s, x, r.s, t);
    r.e = __fadd_rn(a.e, t);
    return r;
  } else {
    return R::op(a, R::load(x));
  }
}

template <class R, class C>
struct GridScanShared {
  PipeShared<C::kNB> pipe;
  typename R::V pre[C::kNB][C::kRows];  // a row's exclusive prefix in its warp
  typename R::V wtot[C::kNB][C::kNW];   // warp totals, then exclusive prefixes in the tile
  typename R::V prefix[C::kNB];
};
template <class R, class C>
constexpr size_t grid_scan_smem() {
  return 1024 + (size_t)C::kNB * C::kTileBytes + sizeof(GridScanShared<R, C>);
}

template <class R, class C, bool PK>
struct GridScanOp {
  using T = typename R::T;
  using V = typename R::V;
  const CUtensorMap *tin, *tout;
  const uint32_t* in;
  uint32_t* out;
  int64_t n, rows;
  uint64_t* agg;
  int excl;
  uint4* bufs;
  GridScanShared<R, C>* sh;
  int64_t cur;  // prefix warps: tiles walked, and their fold
  V run;

  __device__ uint4* buf(int slot) const { return bufs + (size_t)slot * C::kRows * 8; }
  __device__ bool partial(int64_t row) const { return row == rows && rows * 32 < n; }

  __device__ void load(int slot, int64_t tile) const {
    const int64_t r0 = tile * C::kRows;
    uint64_t* bar = sh->pipe.full + slot;
    if (r0 < rows) {
      mbar_arrive_expect_tx(bar, C::kTileBytes);
      tma_load_2d(buf(slot), tin, 0, (int)r0, bar);
    } else {
      mbar_arrive(bar);  // only the partial last row
    }
  }
  __device__ void fold(int slot, int64_t tile) const {
    const int warp = threadIdx.x >> 5, lane = lane_id(), rl = threadIdx.x;
    const int64_t row = tile * C::kRows + rl;
    uint4* b = buf(slot);
    if (partial(row)) {
      const uint32_t pad = to_bits(R::pad());
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const int64_t e = row * 32 + 4 * j;
        uint4 q;
        q.x = e < n ? in[e] : pad;
        q.y = e + 1 < n ? in[e + 1] : pad;
        q.z = e + 2 < n ? in[e + 2] : pad;
        q.w = e + 3 < n ? in[e + 3] : pad;
        b[rl * 8 + (j ^ (rl & 7))] = q;
      }
    }
    V tot = R::ident();
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const uint4 q = b[rl * 8 + (j ^ (rl & 7))];
      tot = op_elem<R>(tot, from_bits<T>(q.x));
      tot = op_elem<R>(tot, from_bits<T>(q.y));
      tot = op_elem<R>(tot, from_bits<T>(q.z));
      tot = op_elem<R>(tot, from_bits<T>(q.w));
    }
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const V u = R::shfl_up(tot, d, 32);
      if (lane >= d) tot = R::op(u, tot);
    }
    const V ex = R::shfl_up(tot, 1, 32);
    sh->pre[slot][rl] = lane == 0 ? R::ident() : ex;
    if (lane == 31) sh->wtot[slot][warp] = tot;
  }
  __device__ void publish(int slot, int64_t tile) const {
    if (lane_id() == 0) {
      V total = R::ident();
#pragma unroll
      for (int k = 0; k < C::kNW; ++k) {
        const V t = sh->wtot[slot][k];
        sh->wtot[slot][k] = total;
        total = R::op(total, t);
      }
      agg_store<R, PK>(agg, tile, total);
    }
  }
  __device__ bool prefix(int slot, int64_t tile, uint32_t limit, volatile int* abort) {
    if (!follow<R, PK>(agg, tile, cur, run, limit, abort)) return false;
    if (lane_id() == 0) sh->prefix[slot] = run;
    return true;
  }
  __device__ void finish(int slot, int64_t tile) const {
    const int rl = threadIdx.x;
    uint4* b = buf(slot);
    V carry = R::op(R::op(sh->prefix[slot], sh->wtot[slot][rl >> 5]), sh->pre[slot][rl]);
    const int64_t row = tile * C::kRows + rl;
    const bool part = partial(row);
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      uint4& s = b[rl * 8 + (j ^ (rl & 7))];
      uint4 q = s;
      uint32_t* w = &q.x;
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const V nx = op_elem<R>(carry, from_bits<T>(w[k]));
        w[k] = to_bits(R::out(excl ? carry : nx));
        carry = nx;
      }
      s = q;
      if (part) {
        const int64_t e = row * 32 + 4 * j;
        if (e < n) out[e] = q.x;
        if (e + 1 < n) out[e + 1] = q.y;
        if (e + 2 < n) out[e + 2] = q.z;
        if (e + 3 < n) out[e + 3] = q.w;
      }
    }
    fence_proxy_async_smem();  // before the bulk store reads the buffer
  }
  __device__ void store(int slot, int64_t tile) const {
    if (tile * C::kRows < rows) {
      tma_store_2d(tout, 0, (int)(tile * C::kRows), buf(slot));
      tma_store_wait_read();
    }
  }
};

template <class R, bool PK>
__global__ void __launch_bounds__(GridCfg<R>::kThreads, 1)
    k_scan_grid_rows(const __grid_constant__ CUtensorMap tin, const __grid_constant__ CUtensorMap tout,
                     const uint32_t* __restrict__ in, uint32_t* __restrict__ out, int64_t n, unsigned* ticket,
                     uint64_t* agg, int64_t ntiles, int excl, uint32_t limit, unsigned* status) {
  using C = GridCfg<R>;
  extern __shared__ uint8_t gsr_raw[];
  uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(gsr_raw) + 1023) & ~uintptr_t(1023));
  GridScanShared<R, C>* sh = reinterpret_cast<GridScanShared<R, C>*>(base + (size_t)C::kNB * C::kTileBytes);
  GridScanOp<R, C, PK> op{&tin, &tout, in, out, n, n / 32, agg, excl, reinterpret_cast<uint4*>(base), sh, 0,
                   R::ident()};
  tile_pipe<C::kNB, C::kNW, 1, C::kFlight>(sh->pipe, op, ntiles, ticket, limit, status);
}

// Short arrays: one tile per CTA in the same three parts, several CTAs per SM
// (tiles go by ticket, so that a CTA only waits for tiles of CTAs that run or
// have run).  The pipeline serves an SM's tiles one after the other, which
// costs about a microsecond each.
//
// The prefix.  32-bit sums take the two-level look-back.  Other values: every
// earlier aggregate read once, by all warps together, from 33 tiles up only
// after the tile before has published: until then most are being written, and
// all CTAs polling all of them made every poll slow.  The wait costs a round
// trip, and with more tiles than are resident an early reader finds most
// aggregates there, so it is left out at both ends.  Time until the last
// prefix, traced on int32 sums of 2^21 / 2^22 / 6 x 10^6 elements: all of them
// polled at once 8.0 / 8.0 / 10.0 us, after the wait 5.6 / 6.9 / 8.1, look-back
// 4.3 / 5.2 / 5.9 (fp32: 8.5 / 7.8 / 9.7 and 5.8 / 6.7 / 8.2; a two-level
// look-back whose group sums are folded in order by the last tile to arrive
// 7.2 / 8.2 / 9.4).  A call of 2^21 int32 sums, inputs in L2: 9.6 us, 13.8 with
// all of them polled at once.
template <class R>
__host__ __device__ constexpr bool is_sum32() {
  return std::is_same<R, Plain<AddU>>::value;
}
struct GridShortCfg {
  static constexpr int kRows = 256, kNB = 1, kNW = kRows / 32;
  static constexpr uint32_t kTileBytes = kRows * 128;
};

template <class R, bool PK>
__global__ void __launch_bounds__(GridShortCfg::kNW * 32)
    k_scan_grid_short(const __grid_constant__ CUtensorMap tin, const __grid_constant__ CUtensorMap tout,
                      const uint32_t* __restrict__ in, uint32_t* __restrict__ out, int64_t n, unsigned* ticket,
                      uint64_t* agg, int64_t ntiles, int excl, int wait, uint32_t limit, unsigned* status) {
  using C = GridShortCfg;
  using V = typename R::V;
  extern __shared__ uint8_t gsr_raw[];
  uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(gsr_raw) + 1023) & ~uintptr_t(1023));
  GridScanShared<R, C>* sh = reinterpret_cast<GridScanShared<R, C>*>(base + C::kTileBytes);
  __shared__ int64_t s_tile;
  __shared__ V s_part[C::kNW];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  GridScanOp<R, C, PK> op{&tin, &tout, in, out, n, n / 32, agg, excl, reinterpret_cast<uint4*>(base), sh, 0,
                      R::ident()};
  if (tid == 0) {
    mbar_init(sh->pipe.full, 1);
    mbar_init_fence();
    const int64_t t = (int64_t)atomicAdd(ticket, 1u);
    op.load(0, t);
    s_tile = t;
  }
  __syncthreads();
  const int64_t tile = s_tile;
  if (__syncthreads_or(!mbar_wait_bounded(sh->pipe.full, 0u, limit))) {
    if (tid == 0) {
      atomicOr(status, (unsigned)kDevTimeout);
      mbar_drain(sh->pipe.full, 0u);
    }
    return;
  }
  op.fold(0, tile);
  __syncthreads();
  if constexpr (is_sum32<R>()) {
    __shared__ int s_bad;
    if (warp == 0) {
      unsigned total = 0;
      if (lane == 0) {
#pragma unroll
        for (int k = 0; k < C::kNW; ++k) {
          const unsigned t = sh->wtot[0][k];
          sh->wtot[0][k] = total;
          total += t;
        }
      }
      total = __shfl_sync(kFull, total, 0);
      const int64_t ngroups = (ntiles + 31) / 32;
      bool gave_up;
      const unsigned prefix =
          look_back_sum2(agg, agg + ntiles, agg + ntiles + ngroups, tile, ntiles, total, limit, status, gave_up);
      if (lane == 0) {
        sh->prefix[0] = prefix;
        s_bad = gave_up;
      }
    }
    __syncthreads();
    if (s_bad) return;
  } else {
    if (warp == 0) op.publish(0, tile);
    V part = R::ident();
    bool ok = true;
    auto wait_for = [&](int64_t t, unsigned ns) {  // its aggregate, bounded
      uint64_t w[2];
      for (uint32_t polls = 0;; ++polls) {
        agg_load<R, PK>(agg, t, w);
        if ((w[0] >> 32) != 0 && (w[1] >> 32) != 0) break;
        if (polls > limit) {
          ok = false;
          break;
        }
        __nanosleep(polls > 64 ? 200 : ns);
      }
      return agg_value<R>(w);
    };
    if (wait) {
      if (tid == 0 && tile > 0) wait_for(tile - 1, 100);
      __syncthreads();
    }
    for (int64_t t = tid; ok && t < tile; t += C::kNW * 32) {
      const V a = wait_for(t, 20);
      part = R::op(part, a);
    }
    __syncwarp();
    part = warp_fold<R>(part);
    if (lane == 0) s_part[warp] = part;
    if (__syncthreads_or(!ok)) {
      if (tid == 0) atomicOr(status, (unsigned)kDevTimeout);
      return;
    }
    if (tid == 0) {
      V p = R::ident();
#pragma unroll
      for (int k = 0; k < C::kNW; ++k) p = R::op(p, s_part[k]);
      sh->prefix[0] = p;
    }
    __syncthreads();
  }
  op.finish(0, tile);
  __syncthreads();
  if (tid == 0) op.store(0, tile);
}

// BLOCK scope, small or unaligned arrays: the CTA is the logical block
// (persistent over blocks).
template <class R>
__global__ void __launch_bounds__(1024) k_scan_block(const uint32_t* __restrict__ in, uint32_t* __restrict__ out,
                                                     int64_t n, int excl) {
  using T = typename R::T;
  using V = typename R::V;
  __shared__ V s_wt[32], s_wp[32];
  const int B = blockDim.x, nw = B >> 5, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int64_t nblk = (n + B - 1) / B;
  for (int64_t lb = blockIdx.x; lb < nblk; lb += gridDim.x) {
    const int64_t i = lb * B + tid;
    V v = R::load(i < n ? from_bits<T>(__ldcs(in + i)) : R::pad());
    {
      const V u = R::shfl_up_fresh(v, 1, 32);
      if (lane >= 1) v = R::op_fresh(u, v);
    }
#pragma unroll
    for (int d = 2; d < 32; d <<= 1) {
      const V u = R::shfl_up(v, d, 32);
      if (lane >= d) v = R::op(u, v);
    }
    if (lane == 31) s_wt[warp] = v;
    __syncthreads();
    if (warp == 0) {  // exclusive scan of the warp totals
      V w = lane < nw ? s_wt[lane] : R::ident();
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const V u = R::shfl_up(w, d, 32);
        if (lane >= d) w = R::op(u, w);
      }
      const V ex = R::shfl_up(w, 1, 32);
      s_wp[lane] = lane == 0 ? R::ident() : ex;
    }
    __syncthreads();
    const V incl = R::op(s_wp[warp], v);
    T y;
    if (!excl) {
      y = R::out(incl);
    } else {
      const V e = R::shfl_up(incl, 1, 32);
      y = R::out(lane == 0 ? s_wp[warp] : e);
    }
    if (i < n) out[i] = to_bits(y);
    __syncthreads();
  }
}

// BLOCK scope over aligned arrays: one row of 32 elements per lane, chunks of
// `rpc` rows (whole logical blocks of rb = B / 32 rows, at most 32 rows) per
// warp through row_ring.  A lane scans its row in registers (scan_row's
// combines: the warp scan of k_scan_block), the block's rows are its rb
// neighbouring lanes, whose totals are scanned by shuffles in the same
// Hillis-Steele order, and every element takes prefix op value: the same
// combines as k_scan_block, hence the same bits, without its three barriers
// per block.  The partial last row (n % 32 elements) is read and written by
// its lane from global memory.
//
// k_scan_block is bound by those barriers (4 bytes per thread between them);
// this kernel by memory, and by issue for compensated sums.  2^26 fp32, B =
// 32 / 256 / 1024: plain 334 / 197 / 225 -> 80 us (6700 GB/s), compensated
// 430 / 280 / 289 -> 97 / 100 / 103 us.  Blocks that leave lanes idle (rpc <
// 32) lose that share: B = 544 (17 rows) 259 -> 95 us plain.  Two chunks per
// warp on three buffers; one chunk on one buffer measured 84 us at B = 256
// plain and 113 us compensated.
constexpr int kBlockScanStages = 3, kBlockScanChunks = 2;
// Smaller arrays are bound by one row's latency, where k_scan_block's warp
// scan ends sooner (its blocks of one warp have to take turns).  us in a graph
// of calls, k_scan_block | rows, plain fp32: B = 256, 2^16 / 2^18 / 2^19
// elements 1.7 | 2.7, 2.3 | 2.7, 3.4 | 2.7; B = 32, 2^16 / 10^5 / 2^18 2.2 |
// 2.6, 2.9 | 2.6, 4.1 | 2.6; compensated, B = 256, 2^19 / 2^20 3.9 | 3.9, 5.8 |
// 3.9.
template <class R>
constexpr int64_t block_rows_min(int block) {
  return R::kComp ? int64_t(1) << 19 : block < 64 ? int64_t(3) << 15 : int64_t(3) << 17;
}

template <class R, bool EXCL>
__global__ void __launch_bounds__(kRingWarps * 32, 2)
    k_scan_block_rows(const __grid_constant__ CUtensorMap tin, const __grid_constant__ CUtensorMap tout,
                      const uint32_t* __restrict__ in, uint32_t* __restrict__ out, int64_t n, int rb, int rpc,
                      uint32_t limit, unsigned* status) {
  using T = typename R::T;
  using V = typename R::V;
  const int lane = threadIdx.x & 31;
  const int pos = lane % rb;  // this lane's row within its logical block
  const int64_t rows = n / 32, all_rows = (n + 31) / 32;
  row_ring<true, kBlockScanStages>(&tin, &tout, rows, (all_rows + rpc - 1) / rpc, rpc, limit, status,
                                         [&](int64_t c, uint4* buf) {
    const int64_t row = c * rpc + lane;
    const bool partial = lane < rpc && row == rows && rows < all_rows;
    uint32_t w[32];
#pragma unroll
    for (int j = 0; j < 8; ++j) {  // unit j of row `lane` sits at unit j ^ (lane & 7)
      const uint4 q = buf[lane * 8 + (j ^ (lane & 7))];
      w[4 * j] = q.x;
      w[4 * j + 1] = q.y;
      w[4 * j + 2] = q.z;
      w[4 * j + 3] = q.w;
    }
    if (partial) {
#pragma unroll
      for (int i = 0; i < 32; ++i) w[i] = row * 32 + i < n ? in[row * 32 + i] : to_bits(R::pad());
    }
    // the row's inclusive scan, its total, and the scan of the block's totals
    uint64_t s[16], e[16];  // compensated: packed pairs
    V v[32];                // otherwise
    V tot;
    if constexpr (R::kComp) {
      float x[32];
#pragma unroll
      for (int i = 0; i < 32; ++i) x[i] = __uint_as_float(w[i]);
      scan_row_pairs<32>(x, s, e);
      float lo;
      f2_unpack(s[15], lo, tot.s);
      f2_unpack(e[15], lo, tot.e);
    } else {
#pragma unroll
      for (int i = 0; i < 32; ++i) v[i] = R::load(from_bits<T>(w[i]));
      scan_row_regs<R, 32>(v);
      tot = v[31];
    }
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      if (d >= rb) break;
      const V u = R::shfl_up(tot, d, 32);
      if (pos >= d) tot = R::op(u, tot);
    }
    const V ex = R::shfl_up(tot, 1, 32);
    const V pre = pos == 0 ? R::ident() : ex;
    // every element: prefix op value (exclusive: the element before)
    if constexpr (R::kComp) {
      const uint64_t ps = f2_pack(pre.s, pre.s), pe = f2_pack(pre.e, pre.e);
      float y[32];
#pragma unroll
      for (int k = 0; k < 16; ++k) {
        uint64_t ns, t;
        f2_two_sum(ps, s[k], ns, t);
        f2_unpack(f2_add(ns, f2_add(f2_add(pe, e[k]), t)), y[2 * k], y[2 * k + 1]);
      }
      if constexpr (EXCL) {
        w[0] = to_bits(R::out(pre));
#pragma unroll
        for (int i = 1; i < 32; ++i) w[i] = __float_as_uint(y[i - 1]);
      } else {
#pragma unroll
        for (int i = 0; i < 32; ++i) w[i] = __float_as_uint(y[i]);
      }
    } else {
      if constexpr (EXCL) {
        w[0] = to_bits(R::out(pre));
#pragma unroll
        for (int i = 1; i < 32; ++i) w[i] = to_bits(R::out(R::op(pre, v[i - 1])));
      } else {
#pragma unroll
        for (int i = 0; i < 32; ++i) w[i] = to_bits(R::out(R::op(pre, v[i])));
      }
    }
    if (partial) {
#pragma unroll
      for (int i = 0; i < 32; ++i)
        if (row * 32 + i < n) out[row * 32 + i] = w[i];
    }
#pragma unroll
    for (int j = 0; j < 8; ++j)
      buf[lane * 8 + (j ^ (lane & 7))] = make_uint4(w[4 * j], w[4 * j + 1], w[4 * j + 2], w[4 * j + 3]);
  });
}

template <class R, bool EXCL>
static cox_status launch_block_rows(const uint32_t* in, uint32_t* out, int64_t n, int block, cudaStream_t st) {
  const int rb = block / 32, rpc = 32 / rb * rb;
  CUtensorMap tin, tout;
  if (!encode_rows32_map(&tin, in, n / 32, rpc) || !encode_rows32_map(&tout, out, n / 32, rpc)) return COX_ECUDA;
  auto k = k_scan_block_rows<R, EXCL>;
  constexpr size_t smem = ring_smem(kBlockScanStages);
  static bool ready[kMaxDevices];  // per device: the kernel may take its shared memory
  bool& rd = ready[device_index()];
  if (!rd) {
    if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
      return COX_ECUDA;
    rd = true;
  }
  const int64_t nch = ((n + 31) / 32 + rpc - 1) / rpc;
  k<<<ring_grid(nch, kBlockScanChunks), kRingWarps * 32, smem, st>>>(tin, tout, in, out, n, rb, rpc,
                                                                          spin_limit(), device_status_word());
  return launch_status();
}

struct ScanWs {
  unsigned* ticket;
  uint32_t* flags;
  uint64_t* agg;
  uint64_t* inc;
};

inline size_t scan_ws_bytes(int64_t ntiles) {
  const size_t f = ((size_t)ntiles * 4 + 255) & ~(size_t)255;
  return kScanWsHeader + f + 2 * (size_t)ntiles * 8;
}

inline ScanWs scan_ws(void* ws, int64_t ntiles) {
  char* p = static_cast<char*>(ws);
  ScanWs w;
  w.ticket = reinterpret_cast<unsigned*>(p);
  w.flags = reinterpret_cast<uint32_t*>(p + kScanWsHeader);
  const size_t f = ((size_t)ntiles * 4 + 255) & ~(size_t)255;
  w.agg = reinterpret_cast<uint64_t*>(p + kScanWsHeader + f);
  w.inc = w.agg + ntiles;
  return w;
}

// Tiles per SM up to which every tile has a CTA of its own (six per SM are
// resident).  A call with inputs in L2 / in memory, short form | pipeline:
// int32 sums of 12 / 16.8 / 18 x 10^6 elements 23.9 | 27.1, 33.6 | 35.3, 36.1 |
// 36.5 us / 28.0 | 28.7, 34.3 | 35.4, 36.5 | 36.7; fp32, which has the dearer
// prefix, 12 x 10^6 27.7 | 27.2 / 32.2 | 28.7, compensated 26.5 | 28.0 / 30.0 |
// 28.9.
template <class R>
constexpr int grid_short_tiles() {
  return is_sum32<R>() ? 16 : 8;
}

// GRID scope over an aligned array of at least one full row.
template <class R, bool PK>
static cox_status launch_grid_rows(const uint32_t* in, uint32_t* out, int64_t n, int excl, void* ws, cudaStream_t st) {
  if (!aligned16(ws)) return COX_EINVAL;
  const int64_t short_tiles = (n + GridShortCfg::kRows * 32 - 1) / (GridShortCfg::kRows * 32);
  const bool use_short = short_tiles <= (int64_t)grid_short_tiles<R>() * sm_count();
  using C = GridCfg<R>;
  const int rows = use_short ? GridShortCfg::kRows : C::kRows;
  const int64_t ntiles = use_short ? short_tiles : (n + C::kRows * 32 - 1) / (C::kRows * 32);
  CUtensorMap tin, tout;
  if (!encode_rows32_map(&tin, in, n / 32, rows) || !encode_rows32_map(&tout, out, n / 32, rows))
    return COX_ECUDA;
  // the ticket, then a zero aggregate per tile, and the look-back's two words
  // per group of tiles (within cox_scan_workspace)
  const size_t words = (size_t)ntiles * agg_words<R, PK>() + (use_short && is_sum32<R>() ? 2 * (size_t)((ntiles + 31) / 32) : 0);
  if (cudaMemsetAsync(ws, 0, kScanWsHeader + words * 8, st) != cudaSuccess) return COX_ECUDA;
  unsigned* ticket = static_cast<unsigned*>(ws);
  uint64_t* agg = reinterpret_cast<uint64_t*>(static_cast<char*>(ws) + kScanWsHeader);
  if (use_short) {
    k_scan_grid_short<R, PK><<<(unsigned)ntiles, GridShortCfg::kNW * 32, grid_scan_smem<R, GridShortCfg>(), st>>>(
        tin, tout, in, out, n, ticket, agg, ntiles, excl, ntiles > 32 && ntiles <= (int64_t)6 * sm_count(),
        spin_limit(), device_status_word());
    return launch_status();
  }
  auto k = k_scan_grid_rows<R, PK>;
  static int grid[kMaxDevices];  // resident CTAs, per device
  int& g = grid[device_index()];
  if (g == 0) {
    if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)grid_scan_smem<R, C>()) !=
        cudaSuccess)
      return COX_ECUDA;
    g = persistent_grid(k, C::kThreads, grid_scan_smem<R, C>(), 1 << 30);
  }
  // (one CTA per SM, and more tiles than all of them have buffers)
  k<<<(unsigned)g, C::kThreads, grid_scan_smem<R, C>(), st>>>(tin, tout, in, out, n, ticket, agg, ntiles, excl,
                                                              spin_limit(), device_status_word());
  return launch_status();
}

template <class R>
static cox_status launch_scan_scope(cox_scope scope, int block, const void* d_in, void* d_out, int64_t n, int excl,
                                    void* ws, size_t ws_bytes, cudaStream_t st) {
  const uint32_t* in = static_cast<const uint32_t*>(d_in);
  uint32_t* out = static_cast<uint32_t*>(d_out);
  if (scope == COX_SCOPE_BLOCK) {
    if (n >= block_rows_min<R>(block) && n / 32 < (int64_t(1) << 31) && aligned16(d_in) && aligned16(d_out))
      return excl ? launch_block_rows<R, true>(in, out, n, block, st) : launch_block_rows<R, false>(in, out, n, block, st);
    auto k = k_scan_block<R>;
    static int gmax[33];
    int& g = gmax[block / 32];
    if (g == 0) g = persistent_grid(k, block, 0, 1 << 30);
    const int64_t nblk = (n + block - 1) / block;
    k<<<(int)(nblk < g ? nblk : g), block, 0, st>>>(in, out, n, excl);
    return launch_status();
  }
  if (n >= 32 && n / 32 < (int64_t(1) << 31) && aligned16(d_in) && aligned16(d_out)) {
    const bool whole = ws_bytes >= cox_scan_workspace(COX_SCOPE_GRID, n);
    if constexpr (R::kComp) {
      // compensated sums also take the workspace of 16384-element tiles (about
      // half of cox_scan_workspace()), with packed aggregates
      const int64_t t = (n + 16383) / 16384;
      if (ws && !whole && ws_bytes >= scan_ws_bytes(t) + 24 * (size_t)((t + 31) / 32))
        return launch_grid_rows<R, true>(in, out, n, excl, ws, st);
    }
    if (!ws || !whole) return COX_ENOMEM;
    return launch_grid_rows<R, false>(in, out, n, excl, ws, st);
  }
  constexpr int TILE = grid_scan_tile<R>();
  const int64_t ntiles = (n + TILE - 1) / TILE;
  if (ntiles > 0xFFFFFFFFll) return COX_EUNSUPPORTED;
  const size_t need = scan_ws_bytes(ntiles);
  if (!ws || ws_bytes < need) return COX_ENOMEM;
  if (!aligned16(ws)) return COX_EINVAL;
  if (cudaMemsetAsync(ws, 0, need, st) != cudaSuccess) return COX_ECUDA;
  const ScanWs w = scan_ws(ws, ntiles);
  auto k = k_scan_grid<R>;
  const size_t smem = (size_t)TILE * 4 * (R::kComp ? 2 : 1) + 16;
  if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
    return COX_ECUDA;
  k<<<(unsigned)ntiles, 256, smem, st>>>(in, out, n, w.ticket, w.flags, w.agg, w.inc, ntiles, excl, spin_limit(),
                                         device_status_word(), aligned16(d_in));
  return launch_status();
}

}  // namespace cox

using namespace cox;

extern "C" size_t cox_scan_workspace(cox_scope scope, int64_t n) {
  if (scope != COX_SCOPE_GRID || n <= 0) return 0;
  const int64_t t = (n + 8191) / 8192;  // enough for every form and tile size
  return scan_ws_bytes(t) + 24 * (size_t)((t + 31) / 32);
}

extern "C" cox_status cox_scan(cox_op op, cox_dtype dt, cox_scope scope, int block_dim, const void* d_in, void* d_out,
                               int64_t n, unsigned flags, int exclusive, void* d_workspace, size_t workspace_bytes,
                               void* stream) {
  if (scope != COX_SCOPE_BLOCK && scope != COX_SCOPE_GRID) return COX_EINVAL;
  if (!valid_block(block_dim) || n < 0 || (exclusive != 0 && exclusive != 1)) return COX_EINVAL;
  if (flags & ~(unsigned)COX_F_COMPENSATED) return COX_EINVAL;
  if (n > 0 && (!d_in || !d_out)) return COX_EINVAL;
  const bool comp = flags & COX_F_COMPENSATED;
  return with_reducer(op, dt, comp, [&](auto r) {
    using R = decltype(r);
    if (n == 0) return COX_OK;
    return launch_scan_scope<R>(scope, block_dim, d_in, d_out, n, exclusive, d_workspace, workspace_bytes,
                                as_stream(stream));
  });
}
