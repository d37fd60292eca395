// Runs of equal keys in sorted rows: one output row per run, in one pass.
//
// The segmented sum behind every canonical result (the distinct (file, word),
// 3-word and pair keys with their counts), the edge deduplication at load and
// the offsets of the ranked index.  A CTA takes the next tile of kRunTile rows
// by an atomic ticket, gives each run head its place in the tile and each
// row the sum of the values before it (one scan over the tile), so that a
// run's sum is the difference between two heads; two bounded look-backs, each
// by one warp, give the output rows before the tile and the part of the run
// open at its start that lies in earlier tiles.  A tile that holds a head
// publishes that second word as final at once, so the look-back normally ends
// at the preceding tile, whatever the length of a run.
//
// fkeys holds (file << 32 | value) per row, or vals the file: rows are equal if key and file are.
//
// Bound by HBM: 12 bytes read per row and 16 written per run.  The former form
// (count heads, scan, write; each head's sum by walking its run) read the rows
// twice and took as long as its longest run.
#include "gt_device.cuh"

namespace gt {
namespace {

constexpr int kRunThreads = 256;
constexpr int kRunItems = 8;  // consecutive rows per thread
constexpr int kRunTile = kRunThreads * kRunItems;
constexpr int kRunWarps = kRunThreads / 32;

template <bool kFile, class K>
__device__ __forceinline__ bool run_head(K k, K prev, uint32_t f, uint32_t prev_f) {
  return k != prev || (kFile && f != prev_f);
}

// What a row carries beside its key.
enum RunRows { kKeyVal, kKeyOnly, kKeyFileVal, kKeyFile, kKeyCode };

// The two flag words of a whole tile, from its rows (by one warp): the number of
// its heads, and the part of the run open at its end that lies in it.
struct TileFlags {
  uint64_t heads, open;
};

template <class K, RunRows kRows>
__device__ __forceinline__ TileFlags run_tile_flags(const K* __restrict__ keys, const uint64_t* __restrict__ fkeys,
                                                 const uint32_t* __restrict__ vals, K key_pad, int64_t tile) {
  constexpr bool kFile = kRows == kKeyFileVal || kRows == kKeyFile;
  constexpr int kShift = kRows == kKeyCode ? kCodeBits : 0;
  const int lane = threadIdx.x & 31;
  uint64_t heads = 0, open = 0;
#pragma unroll 1
  for (int64_t i0 = tile * kRunTile; i0 < (tile + 1) * kRunTile; i0 += 32) {
    const int64_t i = i0 + lane;
    const K k = keys[i] >> kShift, prev = i > 0 ? keys[i - 1] >> kShift : K(0);
    uint32_t f = 0, prev_f = 0, v = 1;
    if (kRows == kKeyVal) v = vals[i];
    if (kRows == kKeyCode) v = code_weight(uint32_t(keys[i]));
    if (kRows == kKeyFileVal) {
      f = uint32_t(fkeys[i] >> 32);
      v = uint32_t(fkeys[i]);
      prev_f = i > 0 ? uint32_t(fkeys[i - 1] >> 32) : 0u;
    }
    if (kRows == kKeyFile) {
      f = vals[i];
      prev_f = i > 0 ? vals[i - 1] : 0u;
    }
    const bool real = k != key_pad;
    const unsigned h = __ballot_sync(0xffffffffu, real && (i == 0 || run_head<kFile>(k, prev, f, prev_f)));
    if (!real) v = 0;
    if (h) {
      heads += unsigned(__popc(h));
      open = lane >= 31 - __clz(h) ? v : 0u;
    } else {
      open += v;
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) open += __shfl_xor_sync(0xffffffffu, open, o);
  return {(tile == 0 ? kFlagIncl : kFlagAgg) | heads, (tile == 0 || heads ? kFlagIncl : kFlagAgg) | open};
}

template <class K, RunRows kRows>
__global__ void __launch_bounds__(kRunThreads) reduce_runs_kernel(
    const K* __restrict__ keys, const uint64_t* __restrict__ fkeys, const uint32_t* __restrict__ vals,
    int64_t n_max, const int64_t* __restrict__ n_dev, K key_pad, const __grid_constant__ RunOut out,
    unsigned long long* __restrict__ look, int64_t tiles_max, int polls) {
  constexpr bool kFile = kRows == kKeyFileVal || kRows == kKeyFile, kVals = kRows == kKeyVal;
  constexpr int kShift = kRows == kKeyCode ? kCodeBits : 0;
  __shared__ K s_key[kRunTile];
  __shared__ uint64_t s_before[kRunTile];  // values of the tile before each head
  __shared__ uint32_t s_file[kFile ? kRunTile : 1];
  __shared__ uint64_t w_sum[kRunWarps];
  __shared__ uint32_t w_heads[kRunWarps];
  __shared__ int64_t s_item, s_prefix, s_carry;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  unsigned long long* const head_flags = look;
  unsigned long long* const open_flags = look + tiles_max;
  if (tid == 0) s_item = int64_t(atomicAdd(look + 2 * tiles_max, 1ull));
  __syncthreads();
  const int64_t n = n_dev ? min(*n_dev, n_max) : n_max;
  const int64_t tiles = (n + kRunTile - 1) / kRunTile;
  const int64_t item = s_item;
  if (item >= tiles) {
    if (tiles == 0 && item == 0 && tid == 0) {
      *out.rows = 0;
      if (out.rows1) *out.rows1 = 1;
      if (out.off) out.off[0] = 0;
    }
    return;
  }
  const int64_t i0 = item * kRunTile + tid * kRunItems;
  K k[kRunItems];
  uint32_t v[kRunItems];
  uint32_t f[kFile ? kRunItems : 1];
  if (i0 + kRunItems <= n) {  // rows are 16-byte aligned (checked by the caller)
    if (sizeof(K) == 8) {
      const ulonglong2* kp = reinterpret_cast<const ulonglong2*>(keys + i0);
#pragma unroll
      for (int j = 0; j < kRunItems / 2; ++j) {
        const ulonglong2 x = kp[j];
        k[2 * j] = K(x.x);
        k[2 * j + 1] = K(x.y);
      }
    } else {
      const uint4* kp = reinterpret_cast<const uint4*>(keys + i0);
#pragma unroll
      for (int j = 0; j < kRunItems / 4; ++j) {
        const uint4 x = kp[j];
        k[4 * j] = K(x.x);
        k[4 * j + 1] = K(x.y);
        k[4 * j + 2] = K(x.z);
        k[4 * j + 3] = K(x.w);
      }
    }
    if (kVals) {
      const uint4* vp = reinterpret_cast<const uint4*>(vals + i0);
#pragma unroll
      for (int j = 0; j < kRunItems / 4; ++j) {
        const uint4 x = vp[j];
        v[4 * j] = x.x;
        v[4 * j + 1] = x.y;
        v[4 * j + 2] = x.z;
        v[4 * j + 3] = x.w;
      }
    }
    if (kRows == kKeyFileVal) {
#pragma unroll
      for (int j = 0; j < kRunItems; ++j) {
        const uint64_t x = fkeys[i0 + j];
        f[j] = uint32_t(x >> 32);
        v[j] = uint32_t(x);
      }
    }
    if (kRows == kKeyFile) {
#pragma unroll
      for (int j = 0; j < kRunItems; ++j) f[j] = vals[i0 + j];
    }
    if (kRows == kKeyCode) {
#pragma unroll
      for (int j = 0; j < kRunItems; ++j) {
        v[j] = code_weight(uint32_t(k[j]));
        k[j] >>= kShift;
      }
    }
  } else {
#pragma unroll
    for (int j = 0; j < kRunItems; ++j) {
      const bool in = i0 + j < n;
      k[j] = in ? keys[i0 + j] : key_pad;
      if (kVals) v[j] = in ? vals[i0 + j] : 0u;
      if (kRows == kKeyFileVal) {
        const uint64_t x = in ? fkeys[i0 + j] : 0;
        f[j] = uint32_t(x >> 32);
        v[j] = uint32_t(x);
      }
      if (kRows == kKeyFile) f[j] = in ? vals[i0 + j] : 0u;
      if (kRows == kKeyCode) {
        v[j] = in ? code_weight(uint32_t(k[j])) : 0u;
        if (in) k[j] >>= kShift;
      }
    }
  }
  // the row before this thread's first one
  K prev = __shfl_up_sync(0xffffffffu, k[kRunItems - 1], 1);
  uint32_t prev_f = kFile ? __shfl_up_sync(0xffffffffu, f[kFile ? kRunItems - 1 : 0], 1) : 0u;
  if (lane == 0 && i0 > 0 && i0 <= n) {
    prev = keys[i0 - 1] >> kShift;
    if (kFile) prev_f = kRows == kKeyFileVal ? uint32_t(fkeys[i0 - 1] >> 32) : vals[i0 - 1];
  }
  uint32_t heads = 0;  // bit j: row j starts a run
  uint64_t sum = 0;
#pragma unroll
  for (int j = 0; j < kRunItems; ++j) {
    const bool real = k[j] != key_pad;
    const bool h = real && ((j == 0 && i0 == 0) || run_head<kFile>(k[j], prev, kFile ? f[kFile ? j : 0] : 0u, prev_f));
    heads |= uint32_t(h) << j;
    if (kRows == kKeyOnly || kRows == kKeyFile) v[j] = 1u;
    if (!real) v[j] = 0u;
    sum += v[j];
    prev = k[j];
    if (kFile) prev_f = f[kFile ? j : 0];
  }
  // exclusive scan of (heads, values) over the tile
  uint32_t hi = __popc(heads);
  uint64_t si = sum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t a = __shfl_up_sync(0xffffffffu, hi, o);
    const uint64_t b = __shfl_up_sync(0xffffffffu, si, o);
    if (lane >= o) {
      hi += a;
      si += b;
    }
  }
  if (lane == 31) {
    w_heads[warp] = hi;
    w_sum[warp] = si;
  }
  __syncthreads();
  uint32_t h_before = hi - __popc(heads), h_total = 0;
  uint64_t s_bef = si - sum, s_total = 0;
#pragma unroll
  for (int w = 0; w < kRunWarps; ++w) {
    if (w < warp) {
      h_before += w_heads[w];
      s_bef += w_sum[w];
    }
    h_total += w_heads[w];
    s_total += w_sum[w];
  }
  if (tid == 0) publish_aggregate(head_flags, item, h_total);
#pragma unroll
  for (int j = 0; j < kRunItems; ++j) {
    if ((heads >> j) & 1u) {
      s_key[h_before] = k[j];
      s_before[h_before] = s_bef;
      if (kFile) s_file[h_before] = f[kFile ? j : 0];
      ++h_before;
    }
    s_bef += v[j];
  }
  __syncthreads();
  if (warp == 0) {
    const int64_t p = warp_look_back(head_flags, item, h_total, nullptr, polls, true, [&](int64_t t) {
      return run_tile_flags<K, kRows>(keys, fkeys, vals, key_pad, t).heads;
    });
    if (lane == 0) s_prefix = p;
  } else if (warp == 1) {
    // values of the open run in earlier tiles; a tile with a head ends the look-back there
    const uint64_t open = h_total ? s_total - s_before[h_total - 1] : s_total;
    if (lane == 0) {
      if (h_total) atomicExch(&open_flags[item], kFlagIncl | open);
      else publish_aggregate(open_flags, item, open);
    }
    __syncwarp();
    const int64_t c = warp_look_back(open_flags, item, open, nullptr, polls, h_total == 0, [&](int64_t t) {
      return run_tile_flags<K, kRows>(keys, fkeys, vals, key_pad, t).open;
    });
    if (lane == 0) s_carry = c;
  }
  __syncthreads();
  const int64_t o0 = s_prefix;
  auto put_sum = [&](int64_t o, uint64_t x) {
    if (out.count) out.count[o] = x;
    if (out.mult) out.mult[o] = uint32_t(x);
    if (out.pay) reinterpret_cast<uint32_t*>(out.pay)[2 * o] = uint32_t(x);
  };
  for (uint32_t r = tid; r < h_total; r += kRunThreads) {
    const uint64_t key = s_key[r];
    const int64_t o = o0 + r;
    if (out.key) out.key[o] = to_output_key(out.low_bits ? key & ((uint64_t(1) << out.low_bits) - 1) : key, out.kb);
    if (out.pay) reinterpret_cast<uint32_t*>(out.pay)[2 * o + 1] = uint32_t(key >> out.low_bits);
    if (out.hi) out.hi[o] = key >> out.low_bits;
    if (out.file) out.file[o] = kFile ? int32_t(s_file[r]) : int32_t(key >> out.low_bits);
    if (out.word) out.word[o] = int32_t(out.low_bits ? key & ((uint64_t(1) << out.low_bits) - 1) : key);
    if (out.off) out.off[o] = item * kRunTile + int64_t(s_before[r]);
    if (r + 1 < h_total) put_sum(o, s_before[r + 1] - s_before[r]);
  }
  if (tid == 0) {
    // the run open at the tile's start ends before its first head; the last tile ends the last run
    if (h_total && o0 > 0) put_sum(o0 - 1, uint64_t(s_carry) + s_before[0]);
    if (item == tiles - 1) {
      const int64_t rows = o0 + h_total;
      if (h_total) put_sum(rows - 1, s_total - s_before[h_total - 1]);
      else if (rows > 0) put_sum(rows - 1, uint64_t(s_carry) + s_total);
      *out.rows = rows;
      if (out.rows1) *out.rows1 = rows + 1;
      if (out.off) out.off[rows] = out.off_end ? *out.off_end : n;
    }
  }
}

}  // namespace

namespace {

template <RunRows kRows, class K>
void launch_runs(gt_ctx* ctx, const K* keys, const uint64_t* fkeys, const uint32_t* vals, int64_t n,
                 const int64_t* n_dev, K key_pad, const RunOut& out, cudaStream_t s) {
  const int64_t tiles = n > 0 ? (n + kRunTile - 1) / kRunTile : 1;
  if ((reinterpret_cast<uintptr_t>(keys) & 15) || (reinterpret_cast<uintptr_t>(vals) & 15))
    fail(GT_EINVAL, "rows to reduce must be 16-byte aligned");
  Buf look(ctx, size_t(2 * tiles + 1) * 8, s);
  GT_CUDA(cudaMemsetAsync(look.p, 0, size_t(2 * tiles + 1) * 8, s));
  reduce_runs_kernel<K, kRows><<<unsigned(tiles), kRunThreads, 0, s>>>(
      keys, fkeys, vals, n, n_dev, key_pad, out, look.as<unsigned long long>(), tiles, look_back_polls());
  GT_LAUNCH_CHECK();
}

}  // namespace

void reduce_runs(gt_ctx* ctx, const uint64_t* keys, const uint64_t* fkeys, const uint32_t* vals, int64_t n,
                 const int64_t* n_dev, uint64_t key_pad, const RunOut& out, cudaStream_t s) {
  if (fkeys) launch_runs<kKeyFileVal>(ctx, keys, fkeys, nullptr, n, n_dev, key_pad, out, s);
  else if (vals) launch_runs<kKeyVal>(ctx, keys, nullptr, vals, n, n_dev, key_pad, out, s);
  else launch_runs<kKeyOnly>(ctx, keys, nullptr, nullptr, n, n_dev, key_pad, out, s);
}

void reduce_runs32(gt_ctx* ctx, const uint32_t* keys, int64_t n, const RunOut& out, cudaStream_t s) {
  launch_runs<kKeyOnly>(ctx, keys, nullptr, nullptr, n, nullptr, ~uint32_t(0), out, s);
}

void reduce_coded_runs(gt_ctx* ctx, const uint64_t* keys, int64_t n, const int64_t* n_dev, const RunOut& out,
                       cudaStream_t s) {
  launch_runs<kKeyCode>(ctx, keys, nullptr, nullptr, n, n_dev, ~uint64_t(0), out, s);
}

void reduce_file_runs(gt_ctx* ctx, const uint64_t* keys, const uint32_t* files, int64_t n, const int64_t* n_dev,
                      const RunOut& out, cudaStream_t s) {
  launch_runs<kKeyFile>(ctx, keys, nullptr, files, n, n_dev, ~uint64_t(0), out, s);
}

void reduce_file_runs(gt_ctx* ctx, const uint32_t* keys, const uint32_t* files, int64_t n, const int64_t* n_dev,
                      const RunOut& out, cudaStream_t s) {
  launch_runs<kKeyFile>(ctx, keys, nullptr, files, n, n_dev, ~uint32_t(0), out, s);
}

}  // namespace gt
