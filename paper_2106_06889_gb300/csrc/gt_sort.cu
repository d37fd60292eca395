// Device primitives: exclusive prefix sum and a stable LSD radix sort.
//
// These back the memory-pool sizing (exclusive scans of per-rule sizes, the
// "memory pool" of Section IV-B), the edge deduplication at load time and the
// canonical ordering of every result.
//
// Both are single-pass kernels: a CTA takes the next tile by an atomic ticket,
// publishes the tile's totals and gets what precedes it by a bounded decoupled
// look-back (see gt_device.cuh); a wait that runs out counts the tile waited for
// from its input instead, so the results are right whatever happened.
#include <algorithm>
#include <type_traits>

#include "gt_device.cuh"

namespace gt {

int look_back_polls() {
  return t_call_ctx ? int(t_call_ctx->param("look_back_polls", kSpinLimit)) : kSpinLimit;
}

namespace {

constexpr int kScanThreads = 256;
constexpr int kScanItems = 8;
constexpr int kScanChunk = kScanThreads * kScanItems;

__device__ __forceinline__ int64_t warp_incl_scan(int64_t v) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    int64_t t = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= o) v += t;
  }
  return v;
}

// Exclusive scan of one value per thread across the block; returns the block
// total through *total.
__device__ __forceinline__ int64_t block_excl_scan(int64_t v, int64_t* total) {
  __shared__ int64_t warp_sums[kScanThreads / 32 + 1];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int64_t incl = warp_incl_scan(v);
  if (lane == 31) warp_sums[warp] = incl;
  __syncthreads();
  if (warp == 0) {
    int64_t w = lane < kScanThreads / 32 ? warp_sums[lane] : 0;
    int64_t wi = warp_incl_scan(w);
    if (lane < kScanThreads / 32) warp_sums[lane] = wi - w;
    if (lane == kScanThreads / 32 - 1) warp_sums[kScanThreads / 32] = wi;  // slot after the last warp
  }
  __syncthreads();
  int64_t r = warp_sums[warp] + incl - v;
  if (total) *total = warp_sums[kScanThreads / 32];
  __syncthreads();
  return r;
}

// The flag word of a whole tile, from its values (by one warp).
__device__ __forceinline__ uint64_t scan_tile_flag(const int64_t* __restrict__ in, int64_t tile) {
  int64_t sum = 0;
#pragma unroll 1
  for (int i = threadIdx.x & 31; i < kScanChunk; i += 32) sum += in[tile * kScanChunk + i];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  return (tile == 0 ? kFlagIncl : kFlagAgg) | uint64_t(sum);
}

// One tile of kScanChunk values per CTA.  With one tile (flags == nullptr) the
// scan starts at 0; otherwise tiles are taken in ticket order (flags[tiles] is
// the ticket) and start at the look-back prefix.  Bound by the 16 bytes per
// value it moves; the former two passes (block sums, then the scan proper, with
// a recursive scan of the sums between them) read the values twice and took
// three to five launches.
__global__ void __launch_bounds__(kScanThreads, 6) scan_kernel(const int64_t* in, int64_t* out, int64_t n,
                                                            unsigned long long* __restrict__ flags, int64_t tiles,
                                                            int polls) {
  __shared__ int64_t tile[kScanChunk];
  __shared__ int64_t s_item, s_prefix;
  int64_t item = 0;
  if (flags) {
    if (threadIdx.x == 0) s_item = int64_t(atomicAdd(&flags[tiles], 1ull));
    __syncthreads();
    item = s_item;
  }
  const int64_t base = item * kScanChunk;
  for (int i = threadIdx.x; i < kScanChunk; i += kScanThreads) {
    const int64_t idx = base + i;
    tile[i] = idx < n ? in[idx] : 0;
  }
  __syncthreads();
  int64_t local[kScanItems];
  int64_t s = 0;
#pragma unroll
  for (int j = 0; j < kScanItems; ++j) {
    local[j] = tile[threadIdx.x * kScanItems + j];
    s += local[j];
  }
  int64_t total;
  int64_t off = block_excl_scan(s, &total);
  if (flags) {
    if (threadIdx.x < 32) {
      if (threadIdx.x == 0) publish_aggregate(flags, item, uint64_t(total));
      __syncwarp();
      const int64_t p = warp_look_back(flags, item, uint64_t(total), nullptr, polls, true,
                                       [&](int64_t t) { return scan_tile_flag(in, t); });
      if (threadIdx.x == 0) s_prefix = p;
    }
    __syncthreads();
    off += s_prefix;
  }
#pragma unroll
  for (int j = 0; j < kScanItems; ++j) {
    tile[threadIdx.x * kScanItems + j] = off;
    off += local[j];
  }
  __syncthreads();
  for (int i = threadIdx.x; i < kScanChunk; i += kScanThreads) {
    const int64_t idx = base + i;
    if (idx < n) out[idx] = tile[i];
  }
}

// ---- radix sort -------------------------------------------------------------
//
// One histogram kernel reads the keys once and counts the digits of every
// pass; each pass is then one scatter kernel whose tiles get their digits'
// first rows by look-back (Adinets & Merrill, "Onesweep: A Faster Least
// Significant Digit Radix Sort for GPUs", arXiv 2206.01784).

constexpr int kRsThreads = 256;  // one thread per digit value in the per-tile bookkeeping
constexpr int kRsWarps = kRsThreads / 32;
constexpr int kRsBins = 256;
constexpr int kRsMaxPasses = 8;
constexpr int kRsSmallItems = 8, kRsLargeItems = 24;  // keys per thread
// Below this many rows tiles of 2048 keys, from there on tiles of 6144: small
// sorts are latency (few tiles), large ones the per-tile bookkeeping over 256
// digits.  Measured for a whole sort (60-bit Zipf keys, 4-byte values), small
// against large tile: 163k rows 77 against 93 us, 700k 111 against 108, 1.4M 157
// against 134, 3.7M 312 against 243, 49M 3379 against 2607.  Tiles of 4096 rows
// take 261 us at 3.7M and 2909 at 49M, of 8192 rows (one CTA less per SM) 9% and
// 14% more than of 6144.
constexpr int64_t kRsLargeRows = int64_t(1) << 20;
// Keys without values: tiles of 8192 rows from here on (64 bits: 1.4M rows 124 us
// against 117 with tiles of 6144, 7.9M 370 against 391, 49M 1941 against 2128).
constexpr int kRsKeyItems = 32;
constexpr int64_t kRsKeyRows = int64_t(1) << 22;

struct RadixPasses {
  int shift[kRsMaxPasses];
  int bits[kRsMaxPasses];
  int n;
};

// Digit counts of every pass in one read of the keys: counts[p * 256 + d].
// Bound by its shared-memory atomics (one per key and pass), and by frequent digits,
// whose atomics in a warp go one after the other: kRhSplit counters per digit, by
// lane, shorten those chains (49M 60-bit keys: 175 -> 152 us).
constexpr int kRhThreads = 512;
constexpr int kRhItems = 4;
constexpr int kRhSplit = 4;

template <class K>
__global__ void __launch_bounds__(kRhThreads) radix_hist_kernel(const K* __restrict__ keys, int64_t n_max,
                                                                const int64_t* __restrict__ n_dev,
                                                                const __grid_constant__ RadixPasses ps,
                                                                unsigned long long* __restrict__ counts) {
  const int64_t n = n_dev ? min(*n_dev, n_max) : n_max;
  __shared__ __align__(16) uint32_t h[kRsMaxPasses * kRsBins * kRhSplit];
  for (int i = threadIdx.x; i < ps.n * kRsBins * kRhSplit; i += kRhThreads) h[i] = 0;
  const uint32_t part = threadIdx.x & (kRhSplit - 1);
  __syncthreads();
  constexpr int64_t kStep = int64_t(kRhThreads) * kRhItems;
  for (int64_t b = blockIdx.x * kStep; b < n; b += gridDim.x * kStep) {
    K k[kRhItems];
#pragma unroll
    for (int j = 0; j < kRhItems; ++j) {
      const int64_t i = b + j * kRhThreads + threadIdx.x;
      k[j] = i < n ? keys[i] : 0;
    }
    for (int p = 0; p < ps.n; ++p) {
      const uint32_t mask = (1u << ps.bits[p]) - 1u;
      const int shift = ps.shift[p];
#pragma unroll
      for (int j = 0; j < kRhItems; ++j)
        if (b + j * kRhThreads + threadIdx.x < n) 
          atomicAdd(&h[(p * kRsBins + (uint32_t(k[j] >> shift) & mask)) * kRhSplit + part], 1u);
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < ps.n * kRsBins; i += kRhThreads) {
    uint32_t c = 0;
#pragma unroll
    for (int q = 0; q < kRhSplit; ++q) c += h[i * kRhSplit + q];
    if (c) atomicAdd(&counts[i], (unsigned long long)(c));
  }
}

// Look-back words of a pass: one per (tile, digit), state in the top two bits
// (1 the tile's own count, 2 the rows of the digit up to and including the
// tile), value below; 32-bit while the rows fit 30 bits, else 64-bit.
template <class W>
struct RsFlag {
  static constexpr W kAgg = W(1) << (sizeof(W) * 8 - 2), kIncl = W(2) << (sizeof(W) * 8 - 2), kVal = kAgg - 1;
};

__device__ __forceinline__ uint32_t ld_relaxed(const uint32_t* p) {
  uint32_t v;
  asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p));
  return v;
}
__device__ __forceinline__ uint64_t ld_relaxed(const uint64_t* p) {
  uint64_t v;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p));
  return v;
}
__device__ __forceinline__ void st_relaxed(uint32_t* p, uint32_t v) {
  asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v));
}
__device__ __forceinline__ void st_relaxed(uint64_t* p, uint64_t v) {
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v));
}

// Rows of one digit in the tiles before `tile`: words are read four tiles at a
// time, nearest first, up to the first one that holds a prefix.  Tiles are
// taken in ticket order, so the ones waited for are running; the wait is
// bounded anyway: after `polls` polls redo(t) gives the word that tile t would
// have published.
template <class W, class Redo>
__device__ __forceinline__ W rs_look_back(const W* __restrict__ words, int64_t tile, int bin, int polls, Redo redo) {
  W sum = 0;
  int64_t t = tile - 1;
  int spins = 0;
  while (true) {
    W v[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) v[q] = t >= q ? ld_relaxed(words + (t - q) * kRsBins + bin) : RsFlag<W>::kIncl;
    int used = 0;
    bool more = true;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      more = more && v[q] > RsFlag<W>::kVal;  // published
      if (more) {
        sum += v[q] & RsFlag<W>::kVal;
        ++used;
        if (v[q] & RsFlag<W>::kIncl) return sum;
      }
    }
    t -= used;
    if (used == 0) {
      if (++spins <= polls) {
        __nanosleep(20);
        continue;
      }
      const W x = redo(t);
      sum += x & RsFlag<W>::kVal;
      if (x & RsFlag<W>::kIncl) return sum;
      --t;
    }
  }
}

// The word of digit `bin` of a whole tile, from its keys (by one thread; tile 0's
// holds the rows of all smaller digits too).
template <class W, class K>
__device__ __forceinline__ W rs_tile_word(const K* __restrict__ kin, int64_t tile, int tile_keys, int shift, uint32_t mask,
                                       uint32_t bin, const unsigned long long* __restrict__ counts) {
  const K* k = kin + tile * tile_keys;
  W c = 0;
#pragma unroll 1
  for (int i = 0; i < tile_keys; ++i) c += (uint32_t(k[i] >> shift) & mask) == bin;
  if (tile != 0) return RsFlag<W>::kAgg | c;
#pragma unroll 1
  for (uint32_t b = 0; b < bin; ++b) c += W(counts[b]);
  return RsFlag<W>::kIncl | c;
}

// Stable scatter of one tile by one digit.  Warp w owns the w-th slice of the
// tile.  The slice's digit counts (one shared atomic per key) give, summed over
// the warps, the tile's counts, published before the keys are ranked; the keys
// are ranked 32 at a time in lane order (one ballot per digit bit) and staged
// in shared memory in digit order, then written with consecutive threads on
// consecutive addresses of each digit's run.
//
// Bound by instruction issue and shared-memory bandwidth rather than HBM: a row
// costs about 25 shared-memory wavefronts per 32 rows (atomic, counter, the
// scattered 8- and 4-byte staging stores, the read back) against the 34 cycles
// its 24 bytes take at the measured copy rate.  The look-back is hidden: with
// every word already published a pass over 49M rows is 6% shorter.  One such pass
// takes 326 us, 173 at the copy rate; of 51M 8-byte keys alone 217 and 120, of 25M
// 4-byte keys alone 85 and 30.
template <class K, int VB, int ITEMS, class W>
__global__ void __launch_bounds__(kRsThreads, ITEMS == kRsSmallItems ? 4 : 2)
    radix_downsweep_kernel(
    const K* __restrict__ kin, K* __restrict__ kout, const void* __restrict__ vin_,
    void* __restrict__ vout_, int64_t n_max, const int64_t* __restrict__ n_dev, int shift, uint32_t mask,
    const unsigned long long* __restrict__ counts, W* __restrict__ words, unsigned* __restrict__ ticket,
    int polls) {
  constexpr int kTileKeys = kRsThreads * ITEMS;
  using VT = typename std::conditional<VB == 8, uint64_t, uint32_t>::type;
  extern __shared__ __align__(16) unsigned char rs_smem[];  // staged keys, then values
  K* skey = reinterpret_cast<K*>(rs_smem);
  VT* sval = reinterpret_cast<VT*>(rs_smem + size_t(kTileKeys) * sizeof(K));
  __shared__ uint32_t wcnt[kRsWarps][kRsBins];
  __shared__ W soff[kRsBins];
  __shared__ W gsum[kRsWarps];
  __shared__ uint32_t wsum[kRsWarps];
  __shared__ unsigned s_tile;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const unsigned lt = (1u << lane) - 1u;
  if (tid == 0) s_tile = atomicAdd(ticket, 1u);
  for (int i = tid; i < kRsWarps * kRsBins; i += kRsThreads) (&wcnt[0][0])[i] = 0;
  __syncthreads();
  const int64_t tile = s_tile;
  const int64_t base = tile * kTileKeys;
  const int64_t n = n_dev ? min(*n_dev, n_max) : n_max;
  if (base >= n) return;  // fewer rows than the grid was sized for; later tiles have none either
  const int tn = int(n - base < kTileKeys ? n - base : kTileKeys);
  const K* kp = kin + base;
  const VT* vp = static_cast<const VT*>(vin_) + (VB ? base : 0);
  const int first = warp * 32 * ITEMS + lane;
  K key[ITEMS];
  VT val[VB ? ITEMS : 1];
  // keys past the end (last tile) count as the top digit and rank after every
  // real key: they stay at the end of the staged tile and are not written
  if (tn == kTileKeys) {
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) key[j] = kp[first + j * 32];
    if (VB) {
#pragma unroll
      for (int j = 0; j < ITEMS; ++j) val[j] = vp[first + j * 32];
    }
  } else {
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) key[j] = first + j * 32 < tn ? kp[first + j * 32] : K(~K(0));
    if (VB) {
#pragma unroll
      for (int j = 0; j < ITEMS; ++j) val[j] = first + j * 32 < tn ? vp[first + j * 32] : VT(0);
    }
  }
  uint32_t* wc = wcnt[warp];
#pragma unroll
  for (int j = 0; j < ITEMS; ++j) atomicAdd(&wc[uint32_t(key[j] >> shift) & mask], 1u);
  __syncthreads();
  // thread = digit: the tile's count, published at once
  uint32_t cnt = 0;
#pragma unroll
  for (int w = 0; w < kRsWarps; ++w) cnt += wcnt[w][tid];
  const uint32_t real = cnt - (uint32_t(tid) == mask ? uint32_t(kTileKeys - tn) : 0u);
  if (tile != 0) st_relaxed(words + tile * kRsBins + tid, RsFlag<W>::kAgg | W(real));
  uint32_t incl = cnt;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += t;
  }
  if (lane == 31) wsum[warp] = incl;
  __syncthreads();
  uint32_t dstart = incl - cnt;
#pragma unroll
  for (int w = 0; w < kRsWarps; ++w) dstart += w < warp ? wsum[w] : 0u;
  {  // each warp's first place of the digit in the staged tile
    uint32_t run = dstart;
#pragma unroll
    for (int w = 0; w < kRsWarps; ++w) {
      const uint32_t c = wcnt[w][tid];
      wcnt[w][tid] = run;
      run += c;
    }
  }
  __syncthreads();
#pragma unroll
  for (int j = 0; j < ITEMS; ++j) {
    const uint32_t d = uint32_t(key[j] >> shift) & mask;
    // 32-bit keys have few passes of narrow digits (18 bits: 3 x 6, 90 -> 85 us over
    // 25M rows); with 64-bit keys and their wider digits the branches cost 0.5% more
    const unsigned peers = warp_digit_peers(d, 0xffffffffu, sizeof(K) == 4 ? mask : 0xffu);
    const uint32_t before = wc[d];
    const uint32_t pos = before + __popc(peers & lt);
    __syncwarp();
    if ((peers & lt) == 0) wc[d] = before + __popc(peers);
    skey[pos] = key[j];
    if (VB) sval[pos] = val[j];
    __syncwarp();
  }
  // the digit's first row: rows of smaller digits, then of earlier tiles
  W excl;
  if (tile == 0) {
    const W c = W(counts[tid]);
    W gi = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const W t = __shfl_up_sync(0xffffffffu, gi, o);
      if (lane >= o) gi += t;
    }
    if (lane == 31) gsum[warp] = gi;
    __syncthreads();
    excl = gi - c;
#pragma unroll
    for (int w = 0; w < kRsWarps; ++w) excl += w < warp ? gsum[w] : W(0);
  } else {
    excl = rs_look_back<W>(words, tile, tid, polls, [&](int64_t t) {
      return rs_tile_word<W, K>(kin, t, kTileKeys, shift, mask, uint32_t(tid), counts);
    });
  }
  st_relaxed(words + tile * kRsBins + tid, RsFlag<W>::kIncl | (excl + real));
  soff[tid] = excl - W(dstart);
  __syncthreads();
  VT* __restrict__ vout = static_cast<VT*>(vout_);
  if (tn == kTileKeys) {
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) {
      const int i = j * kRsThreads + tid;
      const K k = skey[i];
      const W p = soff[uint32_t(k >> shift) & mask] + W(i);
      kout[p] = k;
      if (VB) vout[p] = sval[i];
    }
  } else {
    for (int i = tid; i < tn; i += kRsThreads) {
      const K k = skey[i];
      const W p = soff[uint32_t(k >> shift) & mask] + W(i);
      kout[p] = k;
      if (VB) vout[p] = sval[i];
    }
  }
}

struct RadixScratch {
  unsigned long long* counts;  // [passes * 256]
  unsigned* tickets;           // [passes]
  char* words;                 // [passes][tiles][256]
  size_t zero_bytes;
};

int radix_items(int64_t n, bool keys_only) {
  if (keys_only && n >= kRsKeyRows) return kRsKeyItems;
  const int64_t p = t_call_ctx ? t_call_ctx->param("radix_items", kRsSmallItems) : kRsSmallItems;
  return p == 16 || n >= kRsLargeRows ? kRsLargeItems : kRsSmallItems;
}

// 32-bit look-back words hold fewer than kRsNarrowRows rows; "radix_wide" takes the
// 64-bit ones for up to kRsWideRows rows too
constexpr int64_t kRsNarrowRows = int64_t(1) << 30, kRsWideRows = int64_t(1) << 22;
bool radix_narrow(int64_t n) {
  return n < kRsNarrowRows && !(n <= kRsWideRows && t_call_ctx && t_call_ctx->param("radix_wide", 0));
}

size_t radix_layout(int64_t n, int items, int passes, bool narrow, void* scratch, RadixScratch* out) {
  const int64_t tiles = (n + kRsThreads * items - 1) / (kRsThreads * items);
  const size_t counts = size_t(passes) * kRsBins * 8, tickets = 16 * sizeof(unsigned);
  const size_t words = size_t(passes) * size_t(tiles) * kRsBins * (narrow ? 4 : 8);
  if (out) {
    out->counts = static_cast<unsigned long long*>(scratch);
    out->tickets = reinterpret_cast<unsigned*>(static_cast<char*>(scratch) + counts);
    out->words = static_cast<char*>(scratch) + counts + tickets;
    out->zero_bytes = counts + tickets + words;
  }
  return counts + tickets + words;
}

template <class K, int VB, int ITEMS, class W>
void launch_scatter(const K* ka, K* kb, const void* va, void* vb, int64_t n, const int64_t* n_dev,
                    int shift, uint32_t mask, const RadixScratch& rs, int pass, int polls, cudaStream_t s) {
  constexpr int64_t kTileKeys = int64_t(kRsThreads) * ITEMS;
  constexpr size_t smem = size_t(kTileKeys) * (sizeof(K) + VB);
  const int64_t tiles = (n + kTileKeys - 1) / kTileKeys;
  GT_CUDA(cudaFuncSetAttribute(radix_downsweep_kernel<K, VB, ITEMS, W>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               int(smem)));
  Phase ph(t_call_ctx, "radix_pass", s);  // one span per scatter pass
  radix_downsweep_kernel<K, VB, ITEMS, W><<<unsigned(tiles), kRsThreads, smem, s>>>(
      ka, kb, va, vb, n, n_dev, shift, mask, rs.counts + size_t(pass) * kRsBins,
      reinterpret_cast<W*>(rs.words) + size_t(pass) * size_t(tiles) * kRsBins, rs.tickets + pass, polls);
  GT_LAUNCH_CHECK();
}

template <class K, int VB>
void launch_scatter_any(const K* ka, K* kb, const void* va, void* vb, int64_t n, const int64_t* n_dev,
                        int items, bool narrow, int shift, uint32_t mask, const RadixScratch& rs, int pass, int polls,
                        cudaStream_t s) {
  if (!narrow)
    launch_scatter<K, VB, kRsLargeItems, uint64_t>(ka, kb, va, vb, n, n_dev, shift, mask, rs, pass, polls, s);
  else if (VB == 0 && items == kRsKeyItems)
    launch_scatter<K, VB, VB == 0 ? kRsKeyItems : kRsLargeItems, uint32_t>(
        ka, kb, va, vb, n, n_dev, shift, mask, rs, pass, polls, s);
  else if (items == kRsSmallItems)
    launch_scatter<K, VB, kRsSmallItems, uint32_t>(ka, kb, va, vb, n, n_dev, shift, mask, rs, pass, polls, s);
  else
    launch_scatter<K, VB, kRsLargeItems, uint32_t>(ka, kb, va, vb, n, n_dev, shift, mask, rs, pass, polls, s);
}

// Digit passes over bits [begin_a, end_a) then [begin_b, end_b), the bits of
// each range spread evenly over its passes.
RadixPasses radix_plan(int begin_a, int end_a, int begin_b, int end_b) {
  RadixPasses ps{};
  for (int r = 0; r < 2; ++r) {
    int lo = r ? begin_b : begin_a;
    const int hi = r ? end_b : end_a;
    for (int left = (hi - lo + 7) / 8; left > 0; --left) {
      const int bits = (hi - lo + left - 1) / left;
      if (ps.n == kRsMaxPasses) fail(GT_EINVAL, "more than 64 bits to sort on");
      ps.shift[ps.n] = lo;
      ps.bits[ps.n++] = bits;
      lo += bits;
    }
  }
  return ps;
}

}  // namespace

size_t scan_scratch_bytes(int64_t n) {
  const int64_t nb = (n + kScanChunk - 1) / kScanChunk;
  return nb <= 1 ? 0 : size_t(nb + 1) * sizeof(unsigned long long);
}

void exclusive_scan_i64(const int64_t* in, int64_t* out, int64_t n, void* scratch, cudaStream_t s) {
  if (n <= 0) return;
  const int64_t nb = (n + kScanChunk - 1) / kScanChunk;
  auto* flags = nb > 1 ? static_cast<unsigned long long*>(scratch) : nullptr;
  if (flags) GT_CUDA(cudaMemsetAsync(flags, 0, scan_scratch_bytes(n), s));
  scan_kernel<<<unsigned(nb), kScanThreads, 0, s>>>(in, out, n, flags, nb, look_back_polls());
  GT_LAUNCH_CHECK();
}

size_t radix_scratch_bytes(int64_t n, bool, int) {
  // enough for a sort of any number of rows up to n, whatever "radix_wide" says by
  // then: below kRsLargeRows the tiles are smaller and have more words
  auto bytes = [](int64_t rows, int items, bool narrow) {
    return radix_layout(rows, items, kRsMaxPasses, narrow, nullptr, nullptr);
  };
  const size_t small = bytes(std::min(n, kRsLargeRows - 1), kRsSmallItems, false);
  if (n < kRsLargeRows) return small;
  return std::max({small, bytes(std::min(n, kRsWideRows), kRsLargeItems, false),
                   bytes(n, kRsLargeItems, n < kRsNarrowRows)});
}

namespace {

template <class K>
bool radix_sort_any(K* keys_a, K* keys_b, void* vals_a, void* vals_b, int value_bytes, int64_t n, int begin_a,
                    int end_a, int begin_b, int end_b, void* scratch, cudaStream_t s, const int64_t* n_dev) {
  if (n <= 0) return false;
  const RadixPasses ps = radix_plan(begin_a, end_a, begin_b, end_b);
  if (ps.n == 0) return false;
  const bool narrow = radix_narrow(n);
  const int items = narrow ? radix_items(n, value_bytes == 0) : kRsLargeItems;
  RadixScratch rs;
  radix_layout(n, items, ps.n, narrow, scratch, &rs);
  GT_CUDA(cudaMemsetAsync(scratch, 0, rs.zero_bytes, s));
  const int sms = t_call_ctx ? t_call_ctx->num_sms : 152;
  radix_hist_kernel<K><<<grid_for(n, kRhThreads * kRhItems, sms * 4), kRhThreads, 0, s>>>(keys_a, n, n_dev, ps,
                                                                                                 rs.counts);
  GT_LAUNCH_CHECK();
  const int polls = look_back_polls();
  K *ka = keys_a, *kb = keys_b;
  void *va = vals_a, *vb = vals_b;
  for (int p = 0; p < ps.n; ++p) {
    const uint32_t mask = (1u << ps.bits[p]) - 1u;
    if (value_bytes == 4)
      launch_scatter_any<K, 4>(ka, kb, va, vb, n, n_dev, items, narrow, ps.shift[p], mask, rs, p, polls, s);
    else if (value_bytes == 8)
      launch_scatter_any<K, 8>(ka, kb, va, vb, n, n_dev, items, narrow, ps.shift[p], mask, rs, p, polls, s);
    else
      launch_scatter_any<K, 0>(ka, kb, nullptr, nullptr, n, n_dev, items, narrow, ps.shift[p], mask, rs, p, polls, s);
    std::swap(ka, kb);
    std::swap(va, vb);
  }
  return ps.n % 2 == 1;
}

}  // namespace

bool radix_sort_pingpong(uint64_t* keys_a, uint64_t* keys_b, void* vals_a, void* vals_b, int value_bytes, int64_t n,
                         int begin_a, int end_a, int begin_b, int end_b, void* scratch, cudaStream_t s,
                         const int64_t* n_dev) {
  return radix_sort_any<uint64_t>(keys_a, keys_b, vals_a, vals_b, value_bytes, n, begin_a, end_a, begin_b, end_b,
                                  scratch, s, n_dev);
}

bool radix_sort_pingpong32(uint32_t* keys_a, uint32_t* keys_b, void* vals_a, void* vals_b, int value_bytes, int64_t n,
                           int begin, int end, void* scratch, cudaStream_t s, const int64_t* n_dev) {
  return radix_sort_any<uint32_t>(keys_a, keys_b, vals_a, vals_b, value_bytes, n, begin, end, end, end, scratch, s,
                                  n_dev);
}

void radix_sort_u64(uint64_t* keys_in, uint64_t* keys_out, void* vals_in, void* vals_out, int value_bytes,
                    int64_t n, int begin_bit, int end_bit, void* scratch, cudaStream_t s) {
  radix_sort_u64_split(keys_in, keys_out, vals_in, vals_out, value_bytes, n, begin_bit, end_bit, end_bit, end_bit,
                       scratch, s);
}

void radix_sort_u64_split(uint64_t* keys_in, uint64_t* keys_out, void* vals_in, void* vals_out, int value_bytes,
                          int64_t n, int begin_a, int end_a, int begin_b, int end_b, void* scratch, cudaStream_t s) {
  if (n <= 0) return;
  if (radix_sort_pingpong(keys_in, keys_out, vals_in, vals_out, value_bytes, n, begin_a, end_a, begin_b, end_b,
                          scratch, s))
    return;
  // an even number of passes left the rows in the input buffers
  GT_CUDA(cudaMemcpyAsync(keys_out, keys_in, size_t(n) * 8, cudaMemcpyDeviceToDevice, s));
  if (value_bytes)
    GT_CUDA(cudaMemcpyAsync(vals_out, vals_in, size_t(n) * value_bytes, cudaMemcpyDeviceToDevice, s));
}

}  // namespace gt
