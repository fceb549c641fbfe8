// cox_tile_scan: inclusive scan inside cooperative-groups tiles of width W.
//
// The shuffle scan of the SDK kernel shfl_scan_test (Table 1 of the paper),
// run on a tile: Hillis-Steele steps d = 1, 2, .., W/2 of
//   u = shfl_up(x, d, W); if (rank >= d) x = u op x
// with the lane numbering of Code 3 (element i is global thread i's operand).
// 16-byte aligned arrays take the row-per-lane kernel (k_tile_scan_rows);
// otherwise persistent warps stream chunks of ROWS x 32 elements: 128-bit
// loads, a warp-private shared-memory transpose to one element per lane per
// row, ROWS independent shuffle chains (instruction-level parallelism), and
// the inverse transpose to 128-bit stores.
#include <algorithm>

#include "cox_common.cuh"

namespace cox {

// Rows per warp chunk: plain scans are memory-bound and take 8 rows (two
// 128-bit loads per lane); compensated scans are issue-bound and take 16
// independent rows for instruction-level parallelism (measured ~10% faster at
// width 32 on GB300 than 8 rows with more warps).
template <class R>
constexpr int scan_rows() {
  return R::kComp ? 16 : 8;
}

template <class R, int W, int ROWS>
__global__ void __launch_bounds__(R::kComp ? 256 : 1024) k_tile_scan(const uint32_t* __restrict__ in,
                                                   uint32_t* __restrict__ out, int64_t n, int vec) {
  extern __shared__ uint32_t smem[];
  uint32_t* sm = smem + (threadIdx.x >> 5) * (ROWS * 32);
  constexpr int64_t CH = ROWS * 32;
  const int64_t nchunks = (n + CH - 1) / CH;
  const int64_t wpb = blockDim.x >> 5;
  for (int64_t c = blockIdx.x * wpb + (threadIdx.x >> 5); c < nchunks; c += gridDim.x * wpb)
    scan_chunk<R, W, ROWS>(in, out, n, c, sm, vec != 0);
}

// ------------------------------------------------ one tile row per lane
// (scan_row in cox_common.cuh: each width-W tile collapsed into one
// thread's registers.)

// Warps stream chunks of 32 rows through row_ring: a chunk is read row per
// lane, scanned in registers, written back in place and stored by TMA.
// `n / 32` full rows go through the tensor maps (>= 1 row); the last n % 32
// elements are scanned by thread 0 of CTA 0 from global memory.
//
// Plain scans are bound by memory: one chunk per warp, one buffer (33 KB of
// shared memory per CTA, so other CTAs' loads cover a warp's wait) runs 2^26
// elements at the copy rate (79.6 us; 89.5 us as one persistent wave).
// Compensated scans keep the arithmetic busy for most of that time (16 packed
// adds per element at width 32, two CTAs of 128 registers per thread), so a
// warp takes two chunks with the second in flight under the first's
// arithmetic: widths 4 / 16 / 32 in 79.9 / 80.0 / 81.7 us, against 80.0 /
// 87.8 / 94.5 with one chunk, 80.0 / 82.1 / 90.1 with unpacked adds, and 89.2
// / 94.9 / 89.9 as one persistent wave with unpacked adds.
//
// That is for arrays that stream through memory.  A few chunks per resident
// warp (two CTAs of three buffers per SM) end sooner as one wave of warps that
// stride over the array, whose CTAs start once, most of all with the input in
// L2.  us a call, wave | CTAs from the hardware: plain, width 8, of 2^22 / 2^23
// / 12 x 10^6 elements 6.2 | 7.1, 8.2 | 10.3, 12.0 | 13.5 (input in memory 8.4
// | 8.5, 14.3 | 14.0, 18.5 | 18.2; of 16.8 x 10^6 24.3 | 23.1); compensated,
// width 32, of 2^22 / 2^23 / 2^24 10.3 | 10.3, 12.5 | 14.4, 24.6 | 25.5 (10.6 |
// 12.3, 14.8 | 17.1, 24.8 | 26.4), width 8 of 2^24 20.8 | 22.6 (24.7 | 24.5).
template <class R, int W>
constexpr int rows_wave() {  // chunks per resident warp up to which the wave is taken
  return !R::kComp ? 5 : W >= 16 ? 9 : 7;
}

template <class R, int W, int NS>
__global__ void __launch_bounds__(kRingWarps * 32, 2)
    k_tile_scan_rows(const __grid_constant__ CUtensorMap tin, const __grid_constant__ CUtensorMap tout,
                     const uint32_t* __restrict__ in, uint32_t* __restrict__ out, int64_t n, uint32_t limit,
                     unsigned* status) {
  const int lane = threadIdx.x & 31;
  const int64_t rows = n / 32;
  row_ring<true, NS>(&tin, &tout, rows, (rows + 31) / 32, 32, limit, status, [&](int64_t, uint4* buf) {
    uint32_t w[32];
#pragma unroll
    for (int j = 0; j < 8; ++j) {  // unit j of row `lane` sits at unit j ^ (lane & 7)
      const uint4 q = buf[lane * 8 + (j ^ (lane & 7))];
      w[4 * j] = q.x;
      w[4 * j + 1] = q.y;
      w[4 * j + 2] = q.z;
      w[4 * j + 3] = q.w;
    }
    scan_row<R, W>(w);
#pragma unroll
    for (int j = 0; j < 8; ++j)
      buf[lane * 8 + (j ^ (lane & 7))] = make_uint4(w[4 * j], w[4 * j + 1], w[4 * j + 2], w[4 * j + 3]);
  });
  // The last n % 32 elements: one lane, padded.
  if (blockIdx.x == 0 && threadIdx.x == 0 && rows * 32 < n) {
    const int64_t b = rows * 32;
    const int m = (int)(n - b);
    uint32_t w[32];
#pragma unroll
    for (int i = 0; i < 32; ++i) w[i] = i < m ? in[b + i] : to_bits(R::pad());
    scan_row<R, W>(w);
#pragma unroll
    for (int i = 0; i < 32; ++i)
      if (i < m) out[b + i] = w[i];
  }
}

// One launch over all chunks, `per_warp` of them per warp, or as one wave (0).
template <class R, int W, int NS>
static cox_status launch_rows_as(const void* in, void* out, int64_t n, int per_warp, cudaStream_t st) {
  const int64_t rows = n / 32, nch = (rows + 31) / 32;
  CUtensorMap tin, tout;
  if (!encode_rows32_map(&tin, in, rows, 32) || !encode_rows32_map(&tout, out, rows, 32)) return COX_ECUDA;
  auto k = k_tile_scan_rows<R, W, NS>;
  constexpr size_t smem = ring_smem(NS);
  static int grids[kMaxDevices];  // per device: the resident CTAs
  int& g = grids[device_index()];
  if (g == 0) {
    if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
      return COX_ECUDA;
    g = persistent_grid(k, kRingWarps * 32, smem, 1 << 30);
  }
  const unsigned ctas = per_warp ? ring_grid(nch, per_warp) : std::min(ring_grid(nch, 1), (unsigned)g);
  k<<<ctas, kRingWarps * 32, smem, st>>>(tin, tout, static_cast<const uint32_t*>(in), static_cast<uint32_t*>(out), n,
                                         spin_limit(), device_status_word());
  return launch_status();
}

template <class R, int W>
static cox_status launch_scan_rows(const void* in, void* out, int64_t n, cudaStream_t st) {
  const bool wave = ring_few_chunks((n / 32 + 31) / 32, rows_wave<R, W>());
  if constexpr (R::kComp) return launch_rows_as<R, W, 3>(in, out, n, wave ? 0 : 2, st);
  else return wave ? launch_rows_as<R, W, 3>(in, out, n, 0, st) : launch_rows_as<R, W, 1>(in, out, n, 1, st);
}

template <class R, int W>
static cox_status launch_scan(const void* in, void* out, int64_t n, int block, cudaStream_t st) {
  // Aligned arrays of at least one full row take the row-per-lane kernel; the
  // result does not depend on the CTA size, so block_dim is not needed there.
  if (n >= 32 && n / 32 < (int64_t(1) << 31) && aligned16(in) && aligned16(out))
    return launch_scan_rows<R, W>(in, out, n, st);
  constexpr int kScanRows = scan_rows<R>();
  // The result does not depend on the CTA size; compensated scans run 256-thread
  // CTAs so that their 16 rows of pairs fit in registers.
  if (R::kComp && block > 256) block = 256;
  auto k = k_tile_scan<R, W, kScanRows>;
  const size_t smem = (size_t)(block / 32) * kScanRows * 32 * 4;
  const int64_t chunks = (n + kScanRows * 32 - 1) / (kScanRows * 32);
  const int64_t ctas = (chunks + block / 32 - 1) / (block / 32);
  static int grid_cache[33];  // persistent grid per block size (occupancy does not change)
  int& g = grid_cache[block / 32];
  if (g == 0) g = persistent_grid(k, block, smem, 1 << 30);
  const int grid = (int)(ctas < g ? ctas : g);
  const int vec = aligned16(in) && aligned16(out);
  k<<<grid, block, smem, st>>>(static_cast<const uint32_t*>(in), static_cast<uint32_t*>(out), n, vec);
  return launch_status();
}

}  // namespace cox

using namespace cox;

extern "C" cox_status cox_tile_scan(cox_op op, cox_dtype dt, int width, int block_dim, const void* d_in,
                                    void* d_out, int64_t n, unsigned flags, void* stream) {
  if (!valid_width(width) || !valid_block(block_dim) || n < 0) return COX_EINVAL;
  if (flags & ~(unsigned)COX_F_COMPENSATED) return COX_EINVAL;
  if (n > 0 && (!d_in || !d_out)) return COX_EINVAL;
  const bool comp = flags & COX_F_COMPENSATED;
  return with_reducer(op, dt, comp, [&](auto r) {
    using R = decltype(r);
    return with_width(width, [&](auto w) {
      if (n == 0) return COX_OK;
      return launch_scan<R, decltype(w)::value>(d_in, d_out, n, block_dim, as_stream(stream));
    });
  });
}
