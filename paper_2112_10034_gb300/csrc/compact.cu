// cox_ballot_compact: stable stream compaction from warp ballots.
//
// Tiles of 8192 keys (32 KB) arrive by TMA bulk copies (plain loads for a
// ragged tile) and go through the tile pipeline (tile_pipe.cuh; short arrays:
// one tile per CTA).  In a tile, by eight warps:
//   fold    every warp compacts its 1024 keys in place in one pass
//           (compact_tile.cuh): per row of 32 keys, b = __ballot_sync(keep),
//           rank = kept keys of earlier rows + popc(b & lanemask_lt);
//   publish the scan of the 8 warp counts; the tile's count;
//   prefix  the counts of all earlier tiles;
//   finish  every warp copies its kept keys to out[prefix + offset ..].
#include <mutex>

#include "compact_tile.cuh"
#include "tile_pipe.cuh"

namespace cox {

constexpr int kCompactThreads = 256;
constexpr int kCompactNW = kCompactThreads / 32;
constexpr int kCompactReg = 1024;                            // keys per warp
constexpr int64_t kCompactTile = kCompactNW * kCompactReg;  // 8192 keys
constexpr uint32_t kCompactTileBytes = (uint32_t)kCompactTile * 4;
// Room of a tile in shared memory.  A bulk copy starts and ends on 16-byte
// boundaries: an array that begins `shift` words past one is copied from the
// boundary before the tile to the one after it (words of the neighbouring
// tiles, never beyond the array) and its tile sits `shift` words into the
// buffer.  The first tile, and one whose copy would pass the array's end, are
// loaded word by word.  2^28 keys 4 bytes off, d = 0.1 / 0.5 / 0.9: 256 / 291 /
// 331 us; all tiles loaded word by word in fold, which every later tile waits for, 703 / 751 /
// 789 (577 / 649 / 715 by the cooperative kernel before the pipeline).
constexpr int kCompactBuf = (int)kCompactTile + 4;
// Shape of the pipeline, one CTA per SM: six tiles, two groups of eight worker
// warps, three loads in flight.  2^28 keys at d = 0.1 / 0.5 / 0.9: 246 / 281 /
// 322 us (4800 / 5730 / 6340 GB/s); one group 344 / 367 / 394, three 252 / 283
// / 322 (the workers' passes over the keys, then the tile's way through shared
// memory, bound it).  The cooperative kernel before it, two tiles per CTA and a
// look-back per tile, ran 271 / 326 / 372 us, with this tile body 273 / 327 /
// 371.
constexpr int kCompactNB = 6;      // tiles in shared memory
constexpr int kCompactNG = 2;      // groups of eight worker warps
constexpr int kCompactFlight = 3;  // loads in flight
// Up to this many tiles per SM every tile has a CTA of its own (six fit).  us a
// call at d = 0.5, inputs in L2 (in memory), one tile per CTA | pipeline | the
// cooperative kernel: 10^6 keys 8.2 | 11.2 | 8.3 (9.1 | 12.4 | 9.1), 2^22 13.4 |
// 15.4 | 13.5 (15.4 | 17.3 | 15.9), 2^23 21.5 | 18.6 | 17.5 (22.1 | 19.8 | 20.2),
// 2^24 32.2 | 26.8 | 25.7 (32.5 | 29.2 | 29.1).
constexpr int kCompactShortTiles = 6;
constexpr int kCompactPipeThreads = (kCompactNG * kCompactNW + 3) * 32;

template <int NB>
struct CompactShared {
  PipeShared<NB> pipe;
  uint32_t cnt[NB][kCompactNW];   // a warp's kept keys
  uint32_t off[NB][kCompactNW];   // kept keys of the tile's warps before it
  uint32_t total[NB];
  int64_t prefix[NB];
};

// A published count: flag A (desc_missing tells flags 0 and 3 apart from it).
__device__ __forceinline__ bool count_there(uint64_t d) { return !desc_missing(d); }

// OFF: the array may begin off a 16-byte boundary (compiled in, the offset costs
// 0.5% of an aligned array's time in the pipeline).
template <bool SIGNED, int NB, bool OFF>
struct CompactOp {
  const uint32_t* keys;
  int64_t n;
  LeRule rule;
  uint32_t* out;
  int64_t* d_count;
  uint64_t* desc;
  int64_t ntiles;
  int words_off;  // words of `keys` past a 16-byte boundary
  uint32_t* bufs;
  CompactShared<NB>* sh;
  static constexpr int kWin = 8;  // 32-tile rows per poll of the walk
  int64_t cur = 0, run = 0;  // the prefix warp's walk: tiles passed, and their counts' sum

  __device__ int shift() const { return OFF ? words_off : 0; }
  __device__ uint32_t* buf(int slot) const { return bufs + (size_t)slot * kCompactBuf + shift(); }
  __device__ bool bulk(int64_t tile) const {
    return shift() == 0 ? (tile + 1) * kCompactTile <= n : tile > 0 && (tile + 1) * kCompactTile + 4 - shift() <= n;
  }

  __device__ void load(int slot, int64_t tile) const {
    uint64_t* bar = sh->pipe.full + slot;
    if (bulk(tile)) {
      const uint32_t bytes = kCompactTileBytes + (shift() ? 16u : 0u);
      mbar_arrive_expect_tx(bar, bytes);
      tma_load_1d(buf(slot) - shift(), keys + tile * kCompactTile - shift(), bytes, bar);
    } else {
      mbar_arrive(bar);
    }
  }
  __device__ void fold(int slot, int64_t tile) const {
    const int lane = lane_id(), warp = (threadIdx.x >> 5) % kCompactNW, region = warp * kCompactReg;
    uint32_t* b = buf(slot);
    const int valid = (int)min(kCompactTile, n - tile * kCompactTile);
    if (!bulk(tile)) {
      const uint32_t* src = keys + tile * kCompactTile;
      const int end = min(valid, region + kCompactReg);
      if constexpr (NB == 1 || OFF) {
        // sixteen loads of a lane under way at once: a lone ragged tile is all
        // waiting (1000 keys 8.2 us a call one after the other, 7.0 so), and
        // everything waits for an unaligned array's first (2^24 keys, d = 0.9:
        // 40.1 and 37.6)
#pragma unroll 1
        for (int i0 = region + lane; i0 < end; i0 += 512) {
          uint32_t v[16];
#pragma unroll
          for (int r = 0; r < 16; ++r)
            if (i0 + 32 * r < end) v[r] = src[i0 + 32 * r];
#pragma unroll
          for (int r = 0; r < 16; ++r)
            if (i0 + 32 * r < end) b[i0 + 32 * r] = v[r];
        }
      } else {
        for (int i = region + lane; i < end; i += 32) b[i] = src[i];
      }
      __syncwarp();
    }
    const uint32_t kept =
        compact_region<SIGNED, kCompactReg>(b, region, lane, lanemask_lt(), valid, valid == (int)kCompactTile, rule);
    if (lane == 0) sh->cnt[slot][warp] = kept;
  }
  __device__ void publish(int slot, int64_t tile) const {
    const int lane = lane_id();
    const uint32_t c = lane < kCompactNW ? sh->cnt[slot][lane] : 0u;
    uint32_t incl = c;
#pragma unroll
    for (int d = 1; d < kCompactNW; d <<= 1) {
      const uint32_t u = __shfl_up_sync(kFull, incl, d);
      if (lane >= d) incl += u;
    }
    if (lane < kCompactNW) sh->off[slot][lane] = incl - c;
    if (lane == kCompactNW - 1) {
      sh->total[slot] = incl;
      desc_raise(desc + tile, kFlagA | incl);
    }
  }
  __device__ bool prefix(int slot, int64_t tile, uint32_t limit, volatile int* abort) {
    const int lane = lane_id();
    uint32_t polls = 0;
    while (cur < tile) {
      uint64_t w[kWin];
#pragma unroll
      for (int v = 0; v < kWin; ++v) {
        const int64_t t = cur + v * 32 + lane;
        w[v] = t < tile ? ld_relaxed_u64(desc + t) : 0;
      }
      uint32_t part = 0;
      int step = 0;
#pragma unroll
      for (int v = 0; v < kWin; ++v) {
        if (step != v * 32) break;  // (a gap in an earlier row)
        const unsigned there = __ballot_sync(kFull, count_there(w[v]));
        const int k = there == kFull ? 32 : __ffs(~there) - 1;
        if (lane < k) part += (uint32_t)w[v];
        step += k;
      }
      if (step) {
        run += __reduce_add_sync(kFull, part);
        cur += step;
        polls = 0;
        continue;
      }
      if (++polls > limit || __any_sync(kFull, *abort)) return false;
      __nanosleep(polls > 64 ? 200 : 20);
    }
    if (lane == 0) sh->prefix[slot] = run;
    return true;
  }
  __device__ void finish(int slot, int64_t tile) const {
    const int lane = lane_id(), warp = (threadIdx.x >> 5) % kCompactNW;
    const int64_t prefix = sh->prefix[slot];
    const uint32_t total = sh->total[slot];
    if (prefix + (int64_t)total <= n) {
      uint32_t* dst = out + prefix + sh->off[slot][warp];
      const uint32_t* src = buf(slot) + warp * kCompactReg;
      const int kept = (int)sh->cnt[slot][warp];
#pragma unroll 4
      for (int i = lane; i < kept; i += 32) dst[i] = src[i];
      if (tile == ntiles - 1 && warp == 0 && lane == 0) *d_count = prefix + total;
    }
    fence_proxy_async_smem();  // before the bulk copy that refills the buffer
  }
  __device__ void store(int, int64_t) const {}
};

template <bool SIGNED, bool OFF>
__global__ void __launch_bounds__(kCompactPipeThreads, 1)
    k_ballot_compact(const uint32_t* __restrict__ keys, int64_t n, int64_t thr, uint32_t* __restrict__ out,
                     int64_t* __restrict__ d_count, unsigned* ticket, uint64_t* desc, int64_t ntiles,
                     uint32_t limit, unsigned* status, int shift) {
  extern __shared__ __align__(16) uint32_t smem[];
  auto* sh = reinterpret_cast<CompactShared<kCompactNB>*>(smem + (size_t)kCompactNB * kCompactBuf);
  CompactOp<SIGNED, kCompactNB, OFF> op{keys, n, le_rule<SIGNED>(thr), out, d_count, desc, ntiles, shift, smem, sh};
  tile_pipe<kCompactNB, kCompactNW, kCompactNG, kCompactFlight>(sh->pipe, op, ntiles, ticket, limit, status);
}

// Short arrays, whose tiles are resident at once: one tile per CTA, several
// CTAs per SM, the prefix gathered by all warps together.
template <bool SIGNED>
__global__ void __launch_bounds__(kCompactThreads, 6)
    k_ballot_compact_short(const uint32_t* __restrict__ keys, int64_t n, int64_t thr, uint32_t* __restrict__ out,
                           int64_t* __restrict__ d_count, unsigned* ticket, uint64_t* desc, int64_t ntiles,
                           uint32_t limit, unsigned* status, int shift) {
  extern __shared__ __align__(16) uint32_t smem[];
  auto* sh = reinterpret_cast<CompactShared<1>*>(smem + kCompactBuf);
  __shared__ int64_t s_tile;
  __shared__ uint32_t s_part[kCompactNW];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  CompactOp<SIGNED, 1, true> op{keys, n, le_rule<SIGNED>(thr), out, d_count, desc, ntiles, shift, smem, sh};
  if (tid == 0) {
    mbar_init(sh->pipe.full, 1);
    mbar_init_fence();
    const int64_t t = ntiles > 1 ? (int64_t)atomicAdd(ticket, 1u) : 0;  // (a lone tile saves the round trip)
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
  if (warp == 0) op.publish(0, tile);
  uint32_t part = 0;
  bool ok = true;
  for (int64_t t = tid; ok && t < tile; t += kCompactThreads) {
    uint64_t d;
    for (uint32_t polls = 0; !count_there(d = ld_relaxed_u64(desc + t)); ++polls) {
      if (polls > limit) {
        ok = false;
        break;
      }
      __nanosleep(polls > 64 ? 200 : 20);
    }
    part += (uint32_t)d;
  }
  __syncwarp();
  part = __reduce_add_sync(kFull, part);
  if (lane == 0) s_part[warp] = part;
  if (__syncthreads_or(!ok)) {
    if (tid == 0) atomicOr(status, (unsigned)kDevTimeout);
    return;
  }
  if (tid == 0) {
    int64_t p = 0;
    for (int k = 0; k < kCompactNW; ++k) p += s_part[k];
    sh->prefix[0] = p;
  }
  __syncthreads();
  op.finish(0, tile);
}

}  // namespace cox

using namespace cox;

extern "C" size_t cox_ballot_compact_workspace(int64_t n, int block_dim) {
  if (n < 0 || !valid_block(block_dim)) return 0;
  const int64_t tile = kCompactTile;
  return compact_ws_bytes((n + tile - 1) / tile);
}

extern "C" cox_status cox_ballot_compact(cox_dtype dt, int width, int block_dim, const void* d_keys, int64_t n,
                                         int64_t threshold, void* d_out, int64_t* d_count, void* d_workspace,
                                         size_t workspace_bytes, unsigned flags, void* stream) {
  if (!valid_width(width) || !valid_block(block_dim) || n < 0) return COX_EINVAL;
  if (dt != COX_I32 && dt != COX_U32) return COX_EINVAL;
  if (flags & ~(unsigned)COX_F_WS_READY) return COX_EINVAL;
  if (!d_count || (n > 0 && (!d_keys || !d_out))) return COX_EINVAL;
  cudaStream_t st = as_stream(stream);
  if (n == 0) {
    return cudaMemsetAsync(d_count, 0, sizeof(int64_t), st) == cudaSuccess ? COX_OK : COX_ECUDA;
  }
  const size_t need = cox_ballot_compact_workspace(n, block_dim);
  if (!d_workspace || workspace_bytes < need) return COX_ENOMEM;
  if (!aligned16(d_workspace)) return COX_EINVAL;
  if (!(flags & COX_F_WS_READY) && cudaMemsetAsync(d_workspace, 0, need, st) != cudaSuccess) return COX_ECUDA;
  const int64_t tile = kCompactTile;
  const int64_t ntiles = (n + tile - 1) / tile;
  unsigned* ticket = static_cast<unsigned*>(d_workspace);  // in the header, zero like the descriptors
  uint64_t* desc = reinterpret_cast<uint64_t*>(static_cast<char*>(d_workspace) + kCompactWsHeader);
  const int shift = (int)(reinterpret_cast<uintptr_t>(d_keys) % 16 / 4);
  const uint32_t* keys = static_cast<const uint32_t*>(d_keys);
  uint32_t* outp = static_cast<uint32_t*>(d_out);
  if (ntiles <= (int64_t)kCompactShortTiles * sm_count()) {
    const size_t smem = kCompactBuf * 4 + sizeof(CompactShared<1>);
    auto go = [&](auto kern) {
      kern<<<(unsigned)ntiles, kCompactThreads, smem, st>>>(keys, n, threshold, outp, d_count, ticket, desc, ntiles,
                                                            spin_limit(), device_status_word(), shift);
      return launch_status();
    };
    return dt == COX_I32 ? go(k_ballot_compact_short<true>) : go(k_ballot_compact_short<false>);
  }
  constexpr size_t smem = (size_t)kCompactNB * kCompactBuf * 4 + sizeof(CompactShared<kCompactNB>);
  auto launch = [&](auto kern, int* grid) {
    int& g = grid[device_index()];
    if (g == 0) {
      if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
        return COX_ECUDA;
      g = persistent_grid(kern, kCompactPipeThreads, smem, 1 << 30);
    }
    // (one CTA per SM, and more tiles than all of them have buffers)
    kern<<<(unsigned)g, kCompactPipeThreads, smem, st>>>(keys, n, threshold, outp, d_count, ticket, desc, ntiles,
                                                         spin_limit(), device_status_word(), shift);
    return launch_status();
  };
  static int grid[4][kMaxDevices];  // resident CTAs, per kernel and device
  if (shift)
    return dt == COX_I32 ? launch(k_ballot_compact<true, true>, grid[0]) : launch(k_ballot_compact<false, true>, grid[1]);
  return dt == COX_I32 ? launch(k_ballot_compact<true, false>, grid[2]) : launch(k_ballot_compact<false, false>, grid[3]);
}

// ---------------------------------------------------------------------------
// cox_ballot_compact_static: the same compaction for callers that cannot
// allocate device memory.  Its scratch (the ticket and
// the per-tile descriptors) lives in the fixed array below instead of a
// caller-provided workspace.
//
// The array belongs to the library image: every GPU that loads libcox.so
// holds these bytes until the process exits.  In host code the name
// g_compact_scratch is only a host-side stand-in for the symbol, not a
// device address, so it is never passed to a kernel; the device address is
// looked up with cudaGetSymbolAddress once per device (on that device's first
// call of this entry point, with the device current) and cached.
namespace {

constexpr size_t kStaticScratchBytes = size_t(1) << 20;  // COX_COMPACT_STATIC_SCRATCH_BYTES
static __device__ __align__(256) unsigned char g_compact_scratch[kStaticScratchBytes];

constexpr int kStaticMaxDevices = 64;
void* g_scratch_addr[kStaticMaxDevices];
std::mutex g_scratch_mu;

cox_status static_scratch(void** out) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return COX_ECUDA;
  if (dev < 0 || dev >= kStaticMaxDevices) return COX_EUNSUPPORTED;
  std::lock_guard<std::mutex> g(g_scratch_mu);
  if (!g_scratch_addr[dev]) {
    void* p = nullptr;
    if (cudaGetSymbolAddress(&p, g_compact_scratch) != cudaSuccess || !p) return COX_ECUDA;
    g_scratch_addr[dev] = p;
  }
  *out = g_scratch_addr[dev];
  return COX_OK;
}

}  // namespace

extern "C" cox_status cox_ballot_compact_static(cox_dtype dt, int width, int block_dim, const void* d_keys,
                                                int64_t n, int64_t threshold, void* d_out, int64_t* d_count,
                                                void* stream) {
  if (!valid_width(width) || !valid_block(block_dim) || n < 0) return COX_EINVAL;
  if (dt != COX_I32 && dt != COX_U32) return COX_EINVAL;
  if (!d_count || (n > 0 && (!d_keys || !d_out))) return COX_EINVAL;
  // Larger inputs need more tile descriptors than the fixed scratch holds.
  if (cox_ballot_compact_workspace(n, block_dim) > kStaticScratchBytes) return COX_ENOMEM;
  void* scratch = nullptr;
  const cox_status s = static_scratch(&scratch);
  if (s != COX_OK) return s;
  // The call zeroes the bytes it uses (the descriptors), because the array
  // still holds whatever the previous call left there.
  return cox_ballot_compact(dt, width, block_dim, d_keys, n, threshold, d_out, d_count, scratch,
                            kStaticScratchBytes, 0u, stream);
}
