// sort.cu -- particles into cell order (the sort of Alg. 1 / Alg. 2's
// sort_and_calc_moments step): a stable least-significant-digit radix sort of
// the particles' cell indices, the CSR cell offsets, and the gather of the
// velocities into the sorted order.
//
// Keys are cell indices; an index outside [0, n_cells) becomes n_cells, so
// such particles (left the domain, say) end up behind the last cell and
// belong to no cell.  The key has B = bit_length(n_cells) bits, sorted in
// P = ceil(B / 9) passes of ceil(B / P) bits each (two passes up to 2^18
// cells).  One pass:
//   * radix_hist_kernel: a block counts the digits of four tiles of 4096 keys
//     into counts[digit][tile] (16 bytes of four tiles at once), with one
//     shared-memory atomic a run of equal digits;
//   * scan_tiles_kernel: for every digit the exclusive sum over the tiles, in
//     eight digits a block, written tile by tile (pos[tile][digit], full
//     sectors), and the digit's total;
//   * radix_scatter_kernel: each warp ranks a strip of 512 consecutive keys
//     of the tile stably, 32 at a time, with a per-warp running count per
//     digit; one block-wide step turns the per-warp counts into offsets and
//     the totals into the digits' first positions; the tile is placed sorted
//     by digit in shared memory and each digit's run written to its position,
//     so stores are contiguous runs.
// Ranks only count keys that come earlier in the input, so equal keys keep
// their input order: the result is the stable permutation, the same on
// every run.
// 12M particles nearly in order: 208 us in all with the velocities' gather
// (290 with 512-thread tiles that scanned their digits in one warp, a count
// stored as 4 separate bytes a tile and digit, and three scan kernels a pass;
// the bytes of the passes at the copy rate: 85).  Bound: the scatter by issue
// (41 and 55 us), the histograms and offsets by their loads' latency.
#include <cstdint>

#include "fp_device.cuh"
#include "quads.cuh"

namespace fpc {

constexpr int kSortThreads = 256;
constexpr int kSortWarps = kSortThreads / 32;
constexpr int kSortItems = 16;                         // keys per thread
constexpr int kSortTile = kSortThreads * kSortItems;   // 4096 keys per tile
constexpr int kWarpStrip = kSortTile / kSortWarps;     // 512 consecutive keys per warp
constexpr int kMaxBits = 9;
constexpr int kMaxRadix = 1 << kMaxBits;

constexpr int kHistThreads = 512;
constexpr int kHistTiles = 4;                          // tiles a histogram block counts
constexpr int kScanDigits = 8;                         // digits (warps) a scan block
constexpr int kScanAhead = 4;                          // 16-byte loads a lane has in flight there
constexpr int kScanChunk = 128 * kScanAhead;           // tiles it scans at a time
constexpr int kScanParts = 8;                          // parts of the tiles at most

__device__ __forceinline__ uint32_t cell_key(int32_t c, int64_t n_cells) {  // n_cells < 2^31 - 1
  return min((uint32_t)c, (uint32_t)n_cells);  // (negative: above 2^31)
}

template <bool kFirst>
__global__ void __launch_bounds__(kHistThreads) radix_hist_kernel(const int32_t *__restrict__ cell_of,
                                                                  const uint32_t *__restrict__ keys, int64_t n,
                                                                  int64_t n_cells, int shift, int bits,
                                                                  int64_t tile_stride,
                                                                  uint32_t *__restrict__ counts) {
  grid_wait(cell_of, keys, counts);
  __shared__ uint32_t h[kHistTiles][kMaxRadix];
  const int radix = 1 << bits;
  const uint32_t mask = (uint32_t)(radix - 1);
  for (int d = threadIdx.x; d < kHistTiles * kMaxRadix; d += kHistThreads) h[0][d] = 0u;
  __syncthreads();
  // each warp counts a strip of consecutive keys, four a lane and load; lanes
  // whose four digits agree form runs with their neighbours, and each run
  // adds its length with one shared-memory atomic (cell-ordered input has
  // long runs)
  constexpr int kStrip = kHistTiles * kSortTile / (kHistThreads / 32), kRounds = kStrip / 128;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int64_t s0 = (int64_t)blockIdx.x * (kHistTiles * kSortTile) + (int64_t)w * kStrip;
  uint32_t *hw = h[w * kStrip / kSortTile];
  const uint32_t *src = kFirst ? (const uint32_t *)cell_of : keys;
  const bool vec = ((uintptr_t)src & 15) == 0;
  uint4 x[kRounds];
#pragma unroll
  for (int r = 0; r < kRounds; ++r) {
    const int64_t i = s0 + r * 128 + lane * 4;
    if (vec && i + 4 <= n) {
      x[r] = *reinterpret_cast<const uint4 *>(src + i);
    } else {
      x[r].x = i < n ? src[i] : 0u;
      x[r].y = i + 1 < n ? src[i + 1] : 0u;
      x[r].z = i + 2 < n ? src[i + 2] : 0u;
      x[r].w = i + 3 < n ? src[i + 3] : 0u;
    }
  }
#pragma unroll
  for (int r = 0; r < kRounds; ++r) {
    const int64_t i = s0 + r * 128 + lane * 4;
    uint32_t d[4] = {x[r].x, x[r].y, x[r].z, x[r].w};
#pragma unroll
    for (int k = 0; k < 4; ++k) d[k] = ((kFirst ? cell_key((int32_t)d[k], n_cells) : d[k]) >> shift) & mask;
    const int have = i >= n ? 0 : (n - i < 4 ? (int)(n - i) : 4);
    const bool one = have == 4 && d[0] == d[1] && d[1] == d[2] && d[2] == d[3];
    // a run starts where the left neighbour is not of the same single digit
    const uint32_t tag = one ? d[0] : 0xffffffffu;
    const uint32_t left = __shfl_up_sync(0xffffffffu, tag, 1);
    const unsigned starts = __ballot_sync(0xffffffffu, lane == 0 || !one || left != tag);
    if (one) {
      if ((starts >> lane) & 1u) {
        const unsigned after = lane == 31 ? 0u : starts >> (lane + 1);
        atomicAdd(&hw[d[0]], 4u * (uint32_t)(after ? __ffs(after) : 32 - lane));
      }
    } else {
      uint32_t run = 1;
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        if (k >= have) break;
        if (k + 1 < have && d[k + 1 < 4 ? k + 1 : 3] == d[k]) {
          ++run;
        } else {
          atomicAdd(&hw[d[k]], run);
          run = 1;
        }
      }
    }
  }
  __syncthreads();
  static_assert(kHistTiles == 4, "one 16-byte store a digit");
  for (int d = threadIdx.x; d < radix; d += kHistThreads)
    *reinterpret_cast<uint4 *>(counts + (int64_t)d * tile_stride + (int64_t)blockIdx.x * kHistTiles) =
        make_uint4(h[0][d], h[1][d], h[2][d], h[3][d]);
}

// Warp w of block (x, y) takes digit kScanDigits x + w and the y-th part of
// the tiles (`part` tiles, whole chunks): the exclusive sum of its counts over
// the tiles, starting from the sum of the parts before it, which it adds up
// itself (a few of them: the counts stay in L2), and the digit's total.
__global__ void __launch_bounds__(32 * kScanDigits) scan_tiles_kernel(const uint32_t *__restrict__ counts, int radix,
                                                                      int64_t n_tiles, int64_t tile_stride,
                                                                      int64_t part, uint32_t *__restrict__ pos,
                                                                      uint32_t *__restrict__ totals) {
  grid_wait(counts, pos, totals);
  __shared__ uint32_t out[kScanChunk][kScanDigits + 1];  // [tile][digit]
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int d0 = blockIdx.x * kScanDigits, d = d0 + w;
  const uint4 *row = reinterpret_cast<const uint4 *>(counts + (int64_t)(d < radix ? d : 0) * tile_stride);
  const int64_t vecs = tile_stride / 4, first = blockIdx.y * part;
  const int64_t last = first + part < n_tiles ? first + part : n_tiles;
  uint32_t carry = 0;
#pragma unroll 8
  for (int64_t i = lane; i < first / 4; i += 32) {
    const uint4 y = row[i];
    carry += y.x + y.y + y.z + y.w;
  }
  carry = __reduce_add_sync(0xffffffffu, carry);
  for (int64_t t0 = first; t0 < last; t0 += kScanChunk) {
    uint4 x[kScanAhead];
#pragma unroll
    for (int k = 0; k < kScanAhead; ++k) {
      const int64_t i = t0 / 4 + k * 32 + lane;
      x[k] = d < radix && i < vecs ? row[i] : make_uint4(0u, 0u, 0u, 0u);
    }
    uint32_t inc[kScanAhead];
#pragma unroll
    for (int k = 0; k < kScanAhead; ++k) inc[k] = x[k].x + x[k].y + x[k].z + x[k].w;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1)
#pragma unroll
      for (int k = 0; k < kScanAhead; ++k) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, inc[k], o);
        if (lane >= o) inc[k] += y;
      }
#pragma unroll
    for (int k = 0; k < kScanAhead; ++k) {
      uint32_t run = carry + inc[k] - (x[k].x + x[k].y + x[k].z + x[k].w);
      carry += __shfl_sync(0xffffffffu, inc[k], 31);
      uint32_t(*o)[kScanDigits + 1] = out + k * 128 + lane * 4;
      o[0][w] = run;
      o[1][w] = run += x[k].x;
      o[2][w] = run += x[k].y;
      o[3][w] = run + x[k].z;
    }
    __syncthreads();
    const int nt = (int)(last - t0 < kScanChunk ? last - t0 : kScanChunk);
    const int nd = radix - d0 < kScanDigits ? radix - d0 : kScanDigits;
    for (int i = threadIdx.x; i < nt * kScanDigits; i += 32 * kScanDigits) {
      const int t = i / kScanDigits, k = i % kScanDigits;
      if (k < nd) pos[(t0 + t) * radix + d0 + k] = out[t][k];
    }
    __syncthreads();
  }
  if (d < radix && last == n_tiles && lane == 0) totals[d] = carry;
}

// Lanes of the warp whose digit equals this lane's.  __match_any_sync takes
// some eight cycles a distinct value, a ballot a bit about 60 in all: the
// former for cell-ordered keys (few runs in a warp), the latter for others
// (12M keys, 512 threads a block, us a pass: random order 98 by ballots, 119 by
// match; nearly in order 88 by ballots, 61 by match).
__device__ __forceinline__ unsigned same_digit(uint32_t d, bool valid, int bits, int lane) {
  const uint32_t left = __shfl_up_sync(0xffffffffu, d, 1);
  if (__popc(__ballot_sync(0xffffffffu, lane > 0 && left != d)) <= 8) return __match_any_sync(0xffffffffu, d);
  unsigned peers = __ballot_sync(0xffffffffu, valid);
  if (!valid) peers = ~peers;
  for (int b = 0; b < bits; ++b) {
    const bool one = (d >> b) & 1u;
    const unsigned m = __ballot_sync(0xffffffffu, one);
    peers &= one ? m : ~m;
  }
  return peers;
}

template <bool kFirst>
__global__ void __launch_bounds__(kSortThreads, 4) radix_scatter_kernel(
    const int32_t *__restrict__ cell_of, const uint32_t *__restrict__ keys_in, const int32_t *__restrict__ idx_in,
    int64_t n, int64_t n_cells, int shift, int bits, const uint32_t *__restrict__ pos,
    const uint32_t *__restrict__ totals, uint32_t *__restrict__ keys_out, int32_t *__restrict__ idx_out) {
  grid_wait(cell_of, keys_in, idx_in, pos, totals, keys_out, idx_out);
  // the per-warp digit counts are dead once every key knows its place, so
  // the tile staged sorted by digit reuses their memory
  constexpr int kCountBytes = kSortWarps * kMaxRadix * 2, kStageBytes = kSortTile * 8;
  __shared__ __align__(16) unsigned char raw[kCountBytes > kStageBytes ? kCountBytes : kStageBytes];
  uint16_t(*wc)[kMaxRadix] = reinterpret_cast<uint16_t(*)[kMaxRadix]>(raw);  // per warp: keys of each digit
  uint32_t *sk = reinterpret_cast<uint32_t *>(raw);
  int32_t *si = reinterpret_cast<int32_t *>(raw + kSortTile * 4);
  __shared__ uint32_t lstart[kMaxRadix];  // tile-local start of each digit
  __shared__ int32_t gbase[kMaxRadix];    // output position of the tile's digit d, minus lstart[d]
  __shared__ uint64_t warp_tot[kSortWarps];
  static_assert(2 * kSortThreads == kMaxRadix, "two digits a thread");
  const int radix = 1 << bits;
  const uint32_t mask = (uint32_t)(radix - 1);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  for (int i = threadIdx.x; i < kCountBytes / 16; i += kSortThreads)
    reinterpret_cast<uint4 *>(raw)[i] = make_uint4(0u, 0u, 0u, 0u);
  const int64_t t0 = (int64_t)blockIdx.x * kSortTile;
  const int64_t s0 = t0 + (int64_t)w * kWarpStrip;  // this warp's strip
  uint32_t key[kSortItems];
  int32_t idx[kSortItems];
  uint16_t rank[kSortItems];
#pragma unroll
  for (int r = 0; r < kSortItems; ++r) {  // all loads first
    const int64_t i = s0 + r * 32 + lane;
    key[r] = 0u;
    idx[r] = 0;
    if (i < n) {
      key[r] = kFirst ? (uint32_t)cell_of[i] : keys_in[i];
      if (!kFirst) idx[r] = idx_in[i];
    }
  }
  const int d0 = 2 * threadIdx.x;  // this thread's digits
  uint32_t tile_pos[2] = {0u, 0u}, total[2] = {0u, 0u};
#pragma unroll
  for (int k = 0; k < 2; ++k)
    if (d0 + k < radix) {
      tile_pos[k] = pos[(int64_t)blockIdx.x * radix + d0 + k];
      total[k] = totals[d0 + k];
    }
  __syncthreads();
  if (kFirst) {
#pragma unroll
    for (int r = 0; r < kSortItems; ++r) key[r] = cell_key((int32_t)key[r], n_cells);
  }
  // warp-local stable ranks: key s0 + 32 r + lane comes after every key of
  // rounds < r and after the lanes below it with the same digit
#pragma unroll
  for (int r = 0; r < kSortItems; ++r) {
    const int64_t i = s0 + r * 32 + lane;
    const bool valid = i < n;
    const uint32_t d = valid ? (key[r] >> shift) & mask : (uint32_t)kMaxRadix;
    const unsigned peers = same_digit(d, valid, bits, lane);
    const uint32_t base = valid ? wc[w][d] : 0u;
    __syncwarp();
    if (valid && lane == __ffs(peers) - 1) wc[w][d] = (uint16_t)(base + __popc(peers));
    __syncwarp();
    rank[r] = (uint16_t)(base + __popc(peers & ((1u << lane) - 1u)));
  }
  __syncthreads();
  // per digit (two a thread, their 16-bit counts in one word): the warps'
  // exclusive offsets (in place) and the tile's count; then exclusive sums over
  // the digits of the tile's counts (low word) and of the totals (high word)
  {
    uint32_t run = 0;
#pragma unroll
    for (int q = 0; q < kSortWarps; ++q) {
      uint32_t *c2 = reinterpret_cast<uint32_t *>(&wc[q][d0]);
      const uint32_t c = *c2;
      *c2 = run;
      run += c;
    }
    const uint32_t n0 = run & 0xffffu, n1 = run >> 16;
    const uint64_t x0 = ((uint64_t)total[0] << 32) | n0, x = x0 + (((uint64_t)total[1] << 32) | n1);
    uint64_t inc = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint64_t y = __shfl_up_sync(0xffffffffu, (unsigned long long)inc, o);
      if (lane >= o) inc += y;
    }
    if (lane == 31) warp_tot[w] = inc;
    __syncthreads();
    uint64_t ex = inc - x;
#pragma unroll
    for (int q = 0; q < kSortWarps; ++q) ex += q < w ? warp_tot[q] : 0ull;
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const uint32_t ls = (uint32_t)ex;
      lstart[d0 + k] = ls;
      gbase[d0 + k] = (int32_t)(tile_pos[k] + (uint32_t)(ex >> 32) - ls);
      ex += x0;
    }
  }
  __syncthreads();
  uint32_t lp[kSortItems];
#pragma unroll
  for (int r = 0; r < kSortItems; ++r) {
    const uint32_t d = (key[r] >> shift) & mask;
    lp[r] = lstart[d] + wc[w][d] + rank[r];
  }
  __syncthreads();  // the counts are read; their memory becomes the staging tile
#pragma unroll
  for (int r = 0; r < kSortItems; ++r) {
    const int64_t i = s0 + r * 32 + lane;
    if (i < n) {
      sk[lp[r]] = key[r];
      si[lp[r]] = kFirst ? (int32_t)i : idx[r];
    }
  }
  __syncthreads();
  const int cnt = (int)(n - t0 < kSortTile ? n - t0 : kSortTile);
#pragma unroll
  for (int r = 0; r < kSortItems; ++r) {
    const int k = r * kSortThreads + threadIdx.x;
    if (k >= cnt) break;
    const uint32_t kk = sk[k];
    const uint32_t g = (uint32_t)(gbase[(kk >> shift) & mask] + k);
    if (g < (uint32_t)n) {  // always true for a consistent count / scan; keeps every store in bounds
      keys_out[g] = kk;
      idx_out[g] = si[k];
    }
  }
}

// offsets[c] = first sorted position whose key is >= c, for c in [0, n_cells]:
// position i (0..n, n meaning "past the end" with key n_cells) writes the
// cells after its left neighbour's key up to its own.  A lane takes four
// consecutive positions, kOffItems / 4 times, all loads first.
constexpr int kOffItems = 8;
__global__ void __launch_bounds__(256) cell_offsets_kernel(const uint32_t *__restrict__ keys, int64_t n,
                                                           int64_t n_cells, int64_t *__restrict__ offsets) {
  grid_wait(keys, offsets);
  constexpr int kR = kOffItems / 4;
  const int lane = threadIdx.x & 31;
  const int64_t i0 = (((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * (32 * kOffItems) + 4 * lane;
  if (i0 - 4 * lane > n) return;
  // (keys are at most n_cells, n_cells < 2^31 - 1)
  auto key = [&](int64_t i) -> int32_t { return i >= n ? (int32_t)n_cells : (int32_t)min(keys[i], (uint32_t)n_cells); };
  int32_t cur[kR][4], left = -1;  // left: the key before the warp's first position
  if (i0 - 4 * lane > 0) left = key(i0 - 4 * lane - 1);
#pragma unroll
  for (int j = 0; j < kR; ++j) {
    const int64_t i = i0 + 128 * j;
    if (i + 4 <= n) {
      const uint4 x = *reinterpret_cast<const uint4 *>(keys + i);  // the workspace is aligned
      cur[j][0] = (int32_t)min(x.x, (uint32_t)n_cells), cur[j][1] = (int32_t)min(x.y, (uint32_t)n_cells);
      cur[j][2] = (int32_t)min(x.z, (uint32_t)n_cells), cur[j][3] = (int32_t)min(x.w, (uint32_t)n_cells);
    } else {
#pragma unroll
      for (int u = 0; u < 4; ++u) cur[j][u] = key(i + u);
    }
  }
#pragma unroll
  for (int j = 0; j < kR; ++j) {
    int32_t prev = __shfl_up_sync(0xffffffffu, cur[j][3], 1);
    if (lane == 0) prev = left;
    left = __shfl_sync(0xffffffffu, cur[j][3], 31);
    if (prev == cur[j][3] && prev >= 0) continue;  // keys are sorted: no boundary among the four
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int64_t i = i0 + 128 * j + u;
      if (i <= n)
        for (int32_t c = prev + 1; c <= cur[j][u]; ++c) offsets[c] = i;
      prev = cur[j][u];
    }
  }
}

// v_sorted[d][i] = v[d][perm[i]], four consecutive positions a thread: all
// their loads are in flight together, and stores are 16 bytes where the
// component's alignment allows (69 us for 12M FP32 particles nearly in order
// with a position a thread, 48 now; 336 MB at the copy rate: 49).
template <typename VT>
__global__ void __launch_bounds__(256) gather_sorted_kernel(const VT *__restrict__ v, int64_t n,
                                                            const int32_t *__restrict__ perm, VT *__restrict__ v_sorted,
                                                            int vec) {
  grid_wait(v, perm, v_sorted);
  const int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) * 4;
  if (i >= n) return;
  if (i + 4 <= n) {
    int32_t q[4];
    if (vec & 64) {
      const int4 p = *reinterpret_cast<const int4 *>(perm + i);
      q[0] = p.x, q[1] = p.y, q[2] = p.z, q[3] = p.w;
    } else {
#pragma unroll
      for (int u = 0; u < 4; ++u) q[u] = perm[i + u];
    }
    VT x[3][4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      int64_t p = q[u];
      if (p < 0 || p >= n) p = i + u;  // never taken for a permutation; keeps every load in bounds
#pragma unroll
      for (int d = 0; d < 3; ++d) x[d][u] = v[d * n + p];
    }
#pragma unroll
    for (int d = 0; d < 3; ++d) store_comp(v_sorted + d * n + i, (vec >> (2 * d)) & 3, x[d]);
    return;
  }
  for (int64_t k = i; k < n; ++k) {
    int64_t p = perm[k];
    if (p < 0 || p >= n) p = k;
#pragma unroll
    for (int d = 0; d < 3; ++d) v_sorted[d * n + k] = v[d * n + p];
  }
}

// v_out[d][i] = v[d][i] for i >= *first (the particles behind the last cell)
template <typename VT>
__global__ void __launch_bounds__(256) copy_tail_kernel(const VT *__restrict__ v, VT *__restrict__ v_out, int64_t n,
                                                        const int64_t *__restrict__ first) {
  grid_wait(v, v_out, first);
  const int64_t a = *first;
  for (int64_t i = a + (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    v_out[i] = v[i];
    v_out[n + i] = v[n + i];
    v_out[2 * n + i] = v[2 * n + i];
  }
}

void launch_copy_tail(const void *v, void *v_out, int v_dtype, int64_t n, const int64_t *first, cudaStream_t st) {
  if (n <= 0) return;
  if (v_dtype == FP_V_F32)
    launch_after(copy_tail_kernel<float>, 304, 256, 0, st, (const float *)v, (float *)v_out, n, first);
  else
    launch_after(copy_tail_kernel<double>, 304, 256, 0, st, (const double *)v, (double *)v_out, n, first);
}

static inline size_t sort_align(size_t x) { return (x + 255) & ~(size_t)255; }

struct SortPlan {
  int64_t n_tiles, hist_blocks, tile_stride;
  int passes, bits[4];
  size_t off_keys0, off_keys1, off_idx0, off_idx1, off_counts, off_pos, off_totals, total;
};

static SortPlan sort_plan(int64_t n, int64_t n_cells) {
  SortPlan P{};
  int B = 0;
  while (B < 32 && ((uint64_t)n_cells >> B) != 0) ++B;  // keys are 0..n_cells
  if (B == 0) B = 1;
  P.passes = (B + kMaxBits - 1) / kMaxBits;
  const int per = (B + P.passes - 1) / P.passes;
  int left = B;
  for (int q = 0; q < P.passes; ++q) {
    P.bits[q] = left < per ? left : per;
    left -= P.bits[q];
  }
  P.n_tiles = (n + kSortTile - 1) / kSortTile;
  if (P.n_tiles < 1) P.n_tiles = 1;
  P.hist_blocks = (P.n_tiles + kHistTiles - 1) / kHistTiles;
  P.tile_stride = P.hist_blocks * kHistTiles;
  size_t o = 0;
  auto take = [&](size_t bytes) {
    const size_t at = o;
    o += sort_align(bytes);
    return at;
  };
  P.off_keys0 = take((size_t)n * 4);
  P.off_keys1 = take((size_t)n * 4);
  P.off_idx0 = take((size_t)n * 4);
  P.off_idx1 = take((size_t)n * 4);
  P.off_counts = take((size_t)P.tile_stride * kMaxRadix * 4);
  P.off_pos = take((size_t)P.n_tiles * kMaxRadix * 4);
  P.off_totals = take((size_t)kMaxRadix * 4);
  P.total = o;
  return P;
}

size_t sort_workspace_bytes(int64_t n, int64_t n_cells) { return sort_plan(n, n_cells).total; }

// Sorted keys end in the returned buffer (nullptr on a bad workspace);
// perm (sorted position -> input index) and offsets are written.
void launch_sort_by_cell(const int32_t *cell_of, int64_t n, int64_t n_cells, int32_t *perm, int64_t *offsets,
                         void *ws, cudaStream_t st, const uint32_t **sorted_keys) {
  const SortPlan P = sort_plan(n, n_cells);
  char *w = (char *)ws;
  uint32_t *keys[2] = {(uint32_t *)(w + P.off_keys0), (uint32_t *)(w + P.off_keys1)};
  int32_t *idx[2] = {(int32_t *)(w + P.off_idx0), (int32_t *)(w + P.off_idx1)};
  uint32_t *counts = (uint32_t *)(w + P.off_counts), *pos = (uint32_t *)(w + P.off_pos);
  uint32_t *totals = (uint32_t *)(w + P.off_totals);
  int shift = 0, cur = 0;
  for (int q = 0; q < P.passes; ++q) {
    const int bits = P.bits[q], radix = 1 << bits;
    if (n > 0) {
      if (q == 0)
        launch_after(radix_hist_kernel<true>, (unsigned)P.hist_blocks, kHistThreads, 0, st, cell_of, nullptr, n,
                     n_cells, shift, bits, P.tile_stride, counts);
      else
        launch_after(radix_hist_kernel<false>, (unsigned)P.hist_blocks, kHistThreads, 0, st, nullptr, keys[cur], n,
                     n_cells, shift, bits, P.tile_stride, counts);
      const int64_t chunks = (P.n_tiles + kScanChunk - 1) / kScanChunk;
      const int64_t part = (chunks + kScanParts - 1) / kScanParts * kScanChunk;
      const dim3 grid((unsigned)((radix + kScanDigits - 1) / kScanDigits), (unsigned)((P.n_tiles + part - 1) / part));
      launch_after(scan_tiles_kernel, grid, 32 * kScanDigits, 0, st, counts, radix, P.n_tiles, P.tile_stride, part,
                   pos, totals);
      // the last pass writes the permutation straight into perm
      int32_t *idx_dst = q == P.passes - 1 ? perm : idx[cur ^ 1];
      if (q == 0)
        launch_after(radix_scatter_kernel<true>, (unsigned)P.n_tiles, kSortThreads, 0, st, cell_of, nullptr, nullptr,
                     n, n_cells, shift, bits, pos, totals, keys[cur ^ 1], idx_dst);
      else
        launch_after(radix_scatter_kernel<false>, (unsigned)P.n_tiles, kSortThreads, 0, st, nullptr, keys[cur],
                     idx[cur], n, n_cells, shift, bits, pos, totals, keys[cur ^ 1], idx_dst);
    }
    cur ^= 1;
    shift += bits;
  }
  const int64_t blocks = (n + 1 + 256 * kOffItems - 1) / (256 * kOffItems);
  launch_after(cell_offsets_kernel, (unsigned)blocks, 256, 0, st, keys[cur], n, n_cells, offsets);
  if (sorted_keys) *sorted_keys = keys[cur];
}

void launch_gather_sorted(const void *v, int v_dtype, int64_t n, const int32_t *perm, void *v_sorted,
                          cudaStream_t st) {
  if (n <= 0) return;
  const int64_t blocks = (n + 1023) / 1024;
  const int vec = quad_classes(v_sorted, v_sorted, n, 0, v_dtype == FP_V_F32 ? 4 : 8) |
                  (((uintptr_t)perm & 15) == 0 ? 64 : 0);
  if (v_dtype == FP_V_F32)
    launch_after(gather_sorted_kernel<float>, (unsigned)blocks, 256, 0, st, (const float *)v, n, perm,
                 (float *)v_sorted, vec);
  else
    launch_after(gather_sorted_kernel<double>, (unsigned)blocks, 256, 0, st, (const double *)v, n, perm,
                 (double *)v_sorted, vec);
}

}  // namespace fpc
