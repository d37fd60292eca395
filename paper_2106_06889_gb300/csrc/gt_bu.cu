// Bottom-up per-file analytics (Section IV-A's bottom-up traversal, the
// strategy the paper selects when there are many files, Section V-C).
//
// The paper's bottom-up pass merges every rule's local table into its parents
// and finally merges the tables of the root's children ("level-2 nodes") into
// per-file results.  Here the per-file result is built the same way - root
// words of the file plus, for every distinct (file, root child) pair, the
// child's expansion weighted by how often the file references it - but a
// child's "table" is produced on the fly by walking its derivation depth
// first (an explicit stack bounded by the DAG depth), so no per-rule table has
// to be materialised.  The (file, key, weight) rows are then radix-sorted and
// summed, which yields the canonical order directly.  There is no limit on
// the number of files.
#include <algorithm>

#include "gt_device.cuh"

namespace gt {

int file_strategy(const gt_grammar* g) {
  const int64_t p = gparam(g, "file_strategy", 0);
  if (p == 1 || p == 2) return int(p);
  return g->d.F <= 64 ? 1 : 2;
}

namespace {

constexpr int kMaxStack = 64;

int bits_for(int64_t x) {
  int b = 1;
  while ((int64_t(1) << b) <= x) ++b;
  return b;
}

// Visit the words of expand(c) in order.
template <class Emit>
__device__ __forceinline__ void walk_rule(const DevGrammar& d, int32_t c, Emit&& emit) {
  int64_t spos[kMaxStack], send[kMaxStack];
  int sp = 0;
  int64_t pos = d.rule_off[c], end = d.rule_off[c + 1];
  while (true) {
    if (pos == end) {
      if (sp == 0) return;
      --sp;
      pos = spos[sp];
      end = send[sp];
      continue;
    }
    const int32_t s = d.sym[pos++];
    if (s < d.V) {
      emit(s);
    } else {
      spos[sp] = pos;
      send[sp] = end;
      ++sp;
      const int32_t ch = s - d.V;
      pos = d.rule_off[ch];
      end = d.rule_off[ch + 1];
    }
  }
}

__device__ __forceinline__ int32_t file_of_redge(const DevGrammar& d, int64_t e) {
  return int32_t(upper_bound_dev(d.redge_off, int64_t(d.F) + 1, e) - 1);
}

__global__ void redge_len_kernel(const DevGrammar d, bool windows, int64_t* __restrict__ cnt) {
  for (int64_t e = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; e < d.ER; e += int64_t(gridDim.x) * blockDim.x) {
    const uint64_t l = d.exp_len[d.redge_child[e]];
    cnt[e] = windows ? (l >= 2 ? int64_t(l - 2) : 0) : int64_t(l);
  }
}

// ---- word rows: key = file << kbw | word ----

// Rows of the root's words.  A CTA takes a tile of kRowTile symbols, claims its
// rows with one atomic (rows are sorted next, so their order is free; none is
// spent on a reference) and looks for files only among those the tile spans.
constexpr int kRowThreads = 256;
constexpr int kRowItems = 8;
constexpr int kRowTile = kRowThreads * kRowItems;

// last file f in [lo, hi] that starts at or before position j of the root
__device__ __forceinline__ int32_t file_among(const DevGrammar& d, int32_t lo, int32_t hi, int64_t j) {
  while (lo < hi) {
    const int32_t mid = (lo + hi + 1) >> 1;
    if (d.file_off[mid] <= j) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

__global__ void __launch_bounds__(kRowThreads) root_word_rows_kernel(const DevGrammar d, int kbw,
                                                                     unsigned long long* __restrict__ n,
                                                                     uint64_t* __restrict__ key,
                                                                     uint32_t* __restrict__ val) {
  __shared__ int32_t s_file[2];
  __shared__ uint32_t s_warp[kRowThreads / 32];
  __shared__ unsigned long long s_base;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t j0 = int64_t(blockIdx.x) * kRowTile, j1 = min(d.root_len, j0 + kRowTile);
  if (threadIdx.x < 2) s_file[threadIdx.x] = file_among(d, 0, d.F - 1, threadIdx.x ? j1 - 1 : j0);
  int32_t sy[kRowItems];
  uint32_t c = 0;
#pragma unroll
  for (int k = 0; k < kRowItems; ++k) {
    const int64_t j = j0 + k * kRowThreads + threadIdx.x;
    sy[k] = j < j1 ? d.sym[j] : d.V;
    c += sy[k] < d.V;
  }
  uint32_t incl = c;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += t;
  }
  if (lane == 31) s_warp[warp] = incl;
  __syncthreads();
  uint32_t before = 0, total = 0;
#pragma unroll
  for (int w = 0; w < kRowThreads / 32; ++w) {
    before += w < warp ? s_warp[w] : 0u;
    total += s_warp[w];
  }
  if (threadIdx.x == 0) s_base = total ? atomicAdd(n, (unsigned long long)total) : 0ull;
  __syncthreads();
  // a warp's rows are written 32 symbols at a time, so that its stores are dense
  int64_t o = int64_t(s_base) + before;  // the warp's first row
  const int32_t f_lo = s_file[0], f_hi = s_file[1];
  const unsigned lt = (1u << lane) - 1u;
#pragma unroll
  for (int k = 0; k < kRowItems; ++k) {
    const unsigned words = __ballot_sync(0xffffffffu, sy[k] < d.V);
    if (sy[k] < d.V) {
      const uint64_t f = uint64_t(file_among(d, f_lo, f_hi, j0 + k * kRowThreads + threadIdx.x));
      const int64_t at = o + __popc(words & lt);
      key[at] = (f << kbw) | uint64_t(uint32_t(sy[k]));
      val[at] = 1u;
    }
    o += __popc(words);
  }
}

__global__ void child_word_rows_kernel(const DevGrammar d, int kbw, const int64_t* __restrict__ pos,
                                       uint64_t* __restrict__ key, uint32_t* __restrict__ val) {
  for (int64_t e = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; e < d.ER; e += int64_t(gridDim.x) * blockDim.x) {
    const uint64_t f = uint64_t(file_of_redge(d, e)) << kbw;
    const uint32_t m = d.redge_mult[e];
    int64_t o = pos[e];
    walk_rule(d, d.redge_child[e], [&](int32_t w) {
      key[o] = f | uint64_t(uint32_t(w));
      val[o] = m;
      ++o;
    });
  }
}

// ---- window rows: key = compact 3-word key, file separately ----

// Rows of the windows the root owns: a tile of kTile symbols per CTA, its rows
// claimed with one atomic.
constexpr int kRootWinThreads = kTile / 4;

__global__ void __launch_bounds__(kRootWinThreads) root_window_rows_kernel(const DevGrammar d,
                                                                           const int4* __restrict__ ends, int kb,
                                                                           FileRows out) {
  __shared__ uint32_t s_warp[kRootWinThreads / 32];
  __shared__ unsigned long long s_base;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  TileWin t;
  int32_t file[4];
  tile_windows(d, ends, kb, int64_t(blockIdx.x) * kTile + threadIdx.x * 4, t, file);
  uint32_t c = 0;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    if (t.r[i] != 0) t.n[i] = 0;  // rule bodies in the tile that holds the root's end
    c += t.n[i];
  }
  uint32_t incl = c;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t u = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += u;
  }
  if (lane == 31) s_warp[warp] = incl;
  __syncthreads();
  uint32_t before = incl - c, total = 0;
#pragma unroll
  for (int w = 0; w < kRootWinThreads / 32; ++w) {
    before += w < warp ? s_warp[w] : 0u;
    total += s_warp[w];
  }
  if (threadIdx.x == 0) s_base = total ? atomicAdd(out.n, (unsigned long long)total) : 0ull;
  __syncthreads();
  int64_t o = int64_t(s_base) + before;
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int q = 0; q < 2; ++q)
      if (q < t.n[i]) out.put(o++, file[i], t.k[i][q], 1u);
}

// Rows of every window inside each (file, root child) expansion, from row
// `first` on (pos: exclusive scan of the windows per edge).
__global__ void child_window_rows_kernel(const DevGrammar d, int kb, const int64_t* __restrict__ pos,
                                         const unsigned long long* __restrict__ first, FileRows out) {
  const int64_t base = int64_t(*first);
  for (int64_t e = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; e < d.ER; e += int64_t(gridDim.x) * blockDim.x) {
    const int32_t f = file_of_redge(d, e);
    const uint32_t m = d.redge_mult[e];
    int64_t o = base + pos[e];
    int32_t a = -1, b = -1;
    walk_rule(d, d.redge_child[e], [&](int32_t w) {
      if (a >= 0) out.put(o++, f, pack_compact(a, b, w, kb), m);
      a = b;
      b = w;
    });
  }
}

__global__ void add_rows_kernel(const unsigned long long* __restrict__ first, int64_t more,
                                unsigned long long* __restrict__ n) {
  *n = *first + (unsigned long long)more;
}

// off[f] = first row whose file is >= f (rows sorted by file), f in [0, F].
__global__ void file_offsets_kernel(const int32_t* __restrict__ file, const int64_t* __restrict__ n_dev, int32_t F,
                                    int64_t* __restrict__ off) {
  const int64_t n = *n_dev;
  for (int32_t f = blockIdx.x * blockDim.x + threadIdx.x; f <= F; f += gridDim.x * blockDim.x) {
    int64_t lo = 0, hi = n;
    while (lo < hi) {
      const int64_t mid = (lo + hi) >> 1;
      if (file[mid] < f) lo = mid + 1;
      else hi = mid;
    }
    off[f] = lo;
  }
}

// Inverted index from (file, word) rows: stable sort by word carrying the
// file, so the files come out ascending inside each word; offsets per word.
__global__ void word_keys_kernel(const int32_t* __restrict__ word, const int32_t* __restrict__ file,
                                 const int64_t* __restrict__ n_dev, uint64_t* __restrict__ k,
                                 uint32_t* __restrict__ f) {
  const int64_t n = *n_dev;
  for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < n; i += int64_t(gridDim.x) * blockDim.x) {
    k[i] = uint64_t(uint32_t(word[i]));
    f[i] = uint32_t(file[i]);
  }
}

__global__ void widen_i32_kernel(const int32_t* __restrict__ a, const int64_t* __restrict__ n_dev,
                                 uint64_t* __restrict__ out) {
  const int64_t n = *n_dev;
  for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < n; i += int64_t(gridDim.x) * blockDim.x)
    out[i] = uint64_t(uint32_t(a[i]));
}

__global__ void word_offsets_kernel(const uint64_t* __restrict__ sk, const int64_t* __restrict__ n_dev, int32_t V,
                                    int64_t* __restrict__ off) {
  const int64_t n = *n_dev;
  for (int64_t w = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; w <= V; w += int64_t(gridDim.x) * blockDim.x) {
    int64_t lo = 0, hi = n;
    while (lo < hi) {
      const int64_t mid = (lo + hi) >> 1;
      if (int64_t(sk[mid]) < w) lo = mid + 1;
      else hi = mid;
    }
    off[w] = lo;
  }
}

// ---- small files: expanded and sorted in shared memory, one CTA per file ----
//
// When every file has at most kLocalMax tokens, a CTA expands one file into
// shared memory (root symbols of the file, each rule reference walked), sorts
// its words with an LSD radix sort in shared memory (8-bit digits, ranks by
// ballot multisplit, stable), and run-length encodes them into the file's
// (word, count) rows, written to a slot of the file's length.  A second pass
// packs the slots.  No global sort is involved.

constexpr int kLocalThreads = 256;
constexpr int kLocalWarps = kLocalThreads / 32;
constexpr int64_t kLocalMax = 8192;

// Exclusive prefix over the CTA (kLocalThreads threads); *total gets the sum.
__device__ __forceinline__ int local_scan(int v, int* total, int* warp_tot) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int incl = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int t = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += t;
  }
  if (lane == 31) warp_tot[warp] = incl;
  __syncthreads();
  int before = 0, all = 0;
#pragma unroll
  for (int w = 0; w < kLocalWarps; ++w) {
    const int t = warp_tot[w];
    before += w < warp ? t : 0;
    all += t;
  }
  __syncthreads();
  *total = all;
  return before + incl - v;
}

__device__ __forceinline__ unsigned local_peers(uint32_t dg, unsigned active) {
  unsigned peers = active;
#pragma unroll
  for (int b = 0; b < 8; ++b) {
    const bool bit = (dg >> b) & 1u;
    const unsigned bal = __ballot_sync(0xffffffffu, bit);
    peers &= bit ? bal : ~bal;
  }
  return peers;
}

// Stable LSD radix sort of keys[0, n) over bits [0, key_bits) in shared
// memory, 8-bit digits, ping-ponging between a and b; returns the buffer that
// holds the result.  Warp w ranks its contiguous slice 32 keys at a time.
template <typename K>
__device__ K* local_sort(K* a, K* b, int n, int key_bits, uint32_t (*wcnt)[256], uint32_t* dstart, uint32_t* dtot) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const unsigned lt = (1u << lane) - 1u;
  K* src = a;
  K* dst = b;
  const int per = (n + kLocalWarps * 32 - 1) / (kLocalWarps * 32) * 32;  // warp slice, a multiple of 32
  const int lo = min(n, warp * per), hi = min(n, lo + per);
  for (int shift = 0; shift < key_bits; shift += 8) {
    const uint32_t mask = key_bits - shift >= 8 ? 0xffu : ((1u << (key_bits - shift)) - 1u);
    for (int q = lane; q < 256; q += 32) wcnt[warp][q] = 0;
    __syncwarp();
    for (int i = lo + lane; i < hi; i += 32) atomicAdd(&wcnt[warp][uint32_t(src[i] >> shift) & mask], 1u);
    __syncthreads();
    {  // thread = digit: exclusive over warps, then over digits
      const int dg = tid;
      uint32_t run = 0;
#pragma unroll
      for (int w = 0; w < kLocalWarps; ++w) {
        const uint32_t c = wcnt[w][dg];
        wcnt[w][dg] = run;
        run += c;
      }
      uint32_t incl = run;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
      }
      if (lane == 31) dtot[warp] = incl;
      __syncthreads();
      uint32_t pre = 0;
#pragma unroll
      for (int w = 0; w < kLocalWarps; ++w) pre += w < warp ? dtot[w] : 0u;
      dstart[dg] = pre + incl - run;
    }
    __syncthreads();
    for (int i0 = lo; i0 < hi; i0 += 32) {
      const int i = i0 + lane;
      const bool valid = i < hi;
      const K key = valid ? src[i] : K(0);
      const uint32_t dg = uint32_t(key >> shift) & mask;
      const unsigned peers = local_peers(dg, __ballot_sync(0xffffffffu, valid));
      const uint32_t before = wcnt[warp][dg];
      const uint32_t r = __popc(peers & lt);
      if (valid) dst[dstart[dg] + before + r] = key;
      __syncwarp();
      if (valid && r == 0) wcnt[warp][dg] = before + __popc(peers);
      __syncwarp();
    }
    __syncthreads();
    K* t = src;
    src = dst;
    dst = t;
  }
  return src;
}

// Expand file f into words[0, n) (its root symbols, each reference walked);
// returns n.
__device__ __forceinline__ int local_expand(const DevGrammar& d, int32_t f, uint32_t* words, int* warp_tot) {
  const int tid = threadIdx.x;
  const int64_t r0 = d.file_off[f], r1 = d.file_off[f + 1];
  int base = 0;
  for (int64_t j0 = r0; j0 < r1; j0 += kLocalThreads) {
    const int64_t j = j0 + tid;
    const int32_t sy = j < r1 ? d.sym[j] : 0;
    const int len = j < r1 ? (sy < d.V ? 1 : int(d.exp_len[sy - d.V])) : 0;
    int chunk;
    int o = base + local_scan(len, &chunk, warp_tot);
    if (j < r1) {
      if (sy < d.V) {
        words[o] = uint32_t(sy);
      } else {
        walk_rule(d, sy - d.V, [&](int32_t w) { words[o++] = uint32_t(w); });
      }
    }
    base += chunk;
  }
  __syncthreads();
  return base;
}

// Run-length encoding of sorted keys[0, n): head positions go to heads[];
// returns the number of distinct keys.
template <typename K>
__device__ __forceinline__ int local_heads(const K* keys, int n, uint32_t* heads, int* warp_tot) {
  const int tid = threadIdx.x;
  int rows = 0;
  for (int i0 = 0; i0 < n; i0 += kLocalThreads) {
    const int i = i0 + tid;
    const int head = (i < n && (i == 0 || keys[i] != keys[i - 1])) ? 1 : 0;
    int chunk;
    const int at = rows + local_scan(head, &chunk, warp_tot);
    if (head) heads[at] = uint32_t(i);
    rows += chunk;
  }
  __syncthreads();
  return rows;
}

__global__ void __launch_bounds__(kLocalThreads) local_word_rows_kernel(const DevGrammar d, int cap, int kbw,
                                                                        const int64_t* __restrict__ slot_off,
                                                                        int32_t* __restrict__ slot_word,
                                                                        uint32_t* __restrict__ slot_cnt,
                                                                        int64_t* __restrict__ nrows) {
  extern __shared__ __align__(16) uint32_t lsm[];
  uint32_t* bufa = lsm;
  uint32_t* bufb = lsm + cap;
  __shared__ uint32_t wcnt[kLocalWarps][256];
  __shared__ uint32_t dstart[256];
  __shared__ uint32_t dtot[kLocalWarps];
  __shared__ int warp_tot[kLocalWarps];
  const int tid = threadIdx.x;
  for (int32_t f = blockIdx.x; f < d.F; f += gridDim.x) {
    const int n = local_expand(d, f, bufa, warp_tot);
    uint32_t* src = local_sort(bufa, bufb, n, kbw, wcnt, dstart, dtot);
    uint32_t* dst = src == bufa ? bufb : bufa;
    const int rows = local_heads(src, n, dst, warp_tot);
    const int64_t so = slot_off[f];
    for (int k = tid; k < rows; k += kLocalThreads) {
      const uint32_t a = dst[k], b = k + 1 < rows ? dst[k + 1] : uint32_t(n);
      slot_word[so + k] = int32_t(src[a]);
      slot_cnt[so + k] = b - a;
    }
    if (tid == 0) nrows[f] = rows;
    __syncthreads();
  }
}

// Per-file 3-word windows of small files: the file expanded in shared memory,
// its window keys built and sorted there, one (key, count) row per distinct
// window.  The words alias the second key buffer until the keys are built.
__global__ void __launch_bounds__(kLocalThreads) local_window_rows_kernel(const DevGrammar d, int cap, int kb,
                                                                          int key_bits,
                                                                          const int64_t* __restrict__ slot_off,
                                                                          uint64_t* __restrict__ slot_key,
                                                                          uint32_t* __restrict__ slot_cnt,
                                                                          int64_t* __restrict__ nrows) {
  extern __shared__ __align__(16) uint32_t lsm[];
  uint64_t* ka = reinterpret_cast<uint64_t*>(lsm);
  uint64_t* kz = ka + cap;
  uint32_t* words = reinterpret_cast<uint32_t*>(kz);
  __shared__ uint32_t wcnt[kLocalWarps][256];
  __shared__ uint32_t dstart[256];
  __shared__ uint32_t dtot[kLocalWarps];
  __shared__ int warp_tot[kLocalWarps];
  const int tid = threadIdx.x;
  for (int32_t f = blockIdx.x; f < d.F; f += gridDim.x) {
    const int n = local_expand(d, f, words, warp_tot);
    const int nk = n >= 3 ? n - 2 : 0;
    for (int i = tid; i < nk; i += kLocalThreads)
      ka[i] = pack_compact(int32_t(words[i]), int32_t(words[i + 1]), int32_t(words[i + 2]), kb);
    __syncthreads();
    uint64_t* src = local_sort(ka, kz, nk, key_bits, wcnt, dstart, dtot);
    uint32_t* heads = reinterpret_cast<uint32_t*>(src == ka ? kz : ka);
    const int rows = local_heads(src, nk, heads, warp_tot);
    const int64_t so = slot_off[f];
    for (int k = tid; k < rows; k += kLocalThreads) {
      const uint32_t a = heads[k], b = k + 1 < rows ? heads[k + 1] : uint32_t(nk);
      slot_key[so + k] = src[a];
      slot_cnt[so + k] = b - a;
    }
    if (tid == 0) nrows[f] = rows;
    __syncthreads();
  }
}

// Pack window slots into (key, file, count) rows.
__global__ void local_pack_windows_kernel(int32_t F, const int64_t* __restrict__ slot_off,
                                          const int64_t* __restrict__ row_off, const uint64_t* __restrict__ slot_key,
                                          const uint32_t* __restrict__ slot_cnt, uint64_t* __restrict__ key,
                                          int32_t* __restrict__ file, uint64_t* __restrict__ cnt) {
  const int lane = threadIdx.x & 31;
  const int64_t nwarps = (int64_t(gridDim.x) * blockDim.x) >> 5;
  for (int64_t f = (blockIdx.x * int64_t(blockDim.x) + threadIdx.x) >> 5; f < F; f += nwarps) {
    const int64_t so = slot_off[f], ro = row_off[f], n = row_off[f + 1] - ro;
    for (int64_t k = lane; k < n; k += 32) {
      key[ro + k] = slot_key[so + k];
      file[ro + k] = int32_t(f);
      cnt[ro + k] = slot_cnt[so + k];
    }
  }
}

// Token offsets of the files (slots) from their lengths.
__global__ void file_len_i64_kernel(const uint64_t* __restrict__ len, int32_t F, int64_t* __restrict__ out) {
  for (int32_t f = blockIdx.x * blockDim.x + threadIdx.x; f <= F; f += gridDim.x * blockDim.x)
    out[f] = f < F ? int64_t(len[f]) : 0;
}

// Pack the slots: warp per file.
__global__ void local_pack_kernel(int32_t F, const int64_t* __restrict__ slot_off, const int64_t* __restrict__ row_off,
                                  const int32_t* __restrict__ slot_word, const uint32_t* __restrict__ slot_cnt,
                                  int32_t* __restrict__ word, int32_t* __restrict__ file, uint64_t* __restrict__ cnt) {
  const int lane = threadIdx.x & 31;
  const int64_t nwarps = (int64_t(gridDim.x) * blockDim.x) >> 5;
  for (int64_t f = (blockIdx.x * int64_t(blockDim.x) + threadIdx.x) >> 5; f < F; f += nwarps) {
    const int64_t so = slot_off[f], ro = row_off[f], n = row_off[f + 1] - ro;
    for (int64_t k = lane; k < n; k += 32) {
      word[ro + k] = slot_word[so + k];
      file[ro + k] = int32_t(f);
      cnt[ro + k] = slot_cnt[so + k];
    }
  }
}

// ---- the files' words, expanded --------------------------------------------------

// last file f in [lo, hi] whose first word is at or before position p
__device__ __forceinline__ int32_t file_from(const int64_t* __restrict__ first, int32_t lo, int32_t hi, int64_t p) {
  while (lo < hi) {
    const int32_t mid = (lo + hi + 1) >> 1;
    if (first[mid] <= p) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

// words[0, N): the expansion of the root, files back to back.  A tile of kRowTile
// root symbols per CTA in ticket order, kRowItems consecutive ones per thread; a
// tile's first word comes from a bounded look-back over the tiles' lengths.  The
// first kExpandWords words of a tile pass through shared memory, so that they are
// written dense (a thread's words are consecutive: direct stores touch a sector
// per lane); a tile that expands further writes the rest from its threads.
// The references that fit are listed first and walked by all threads in turn, each
// at its place in the stage, which holds the rule till then: bound by the latency of
// the walks (dependent loads of short rule bodies), and a thread's own references
// one after the other made the longest chain.
//
// ends (or null): the rules' first and last two words; they are all of a rule of up
// to four words, which then is one 16-byte load instead of a walk.
//
// file_bits >= 0: words[p] is word << file_bits | file instead.
constexpr int kExpandWords = 6 * 1024;

// From this many root symbols on the ends are worked out first: they take a pass
// over all rules and its launches.  Term vector and index of many files, us, by
// walking every reference / with the ends: 0.7M root symbols 399 / 414, 2.5M 504 /
// 515, 5.6M 600 / 614, 8.2M 733 / 738, 10.8M 862 / 861, 13.4M 998 / 988, 16.6M
// 1170 / 1135 (the expansion itself 253 / 188, the ends 36).
constexpr int64_t kExpandEnds = int64_t(12) << 20;

// The flag word of a whole tile, from its symbols (by one warp).
__device__ __forceinline__ uint64_t expand_tile_flag(const int32_t* __restrict__ sym, const uint64_t* __restrict__ exp_len,
                                                  int32_t V, int64_t tile) {
  int64_t len = 0;
#pragma unroll 1
  for (int i = threadIdx.x & 31; i < kRowTile; i += 32) {
    const int32_t sy = sym[tile * kRowTile + i];
    len += sy < V ? 1 : int64_t(exp_len[sy - V]);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) len += __shfl_xor_sync(0xffffffffu, len, o);
  return (tile == 0 ? kFlagIncl : kFlagAgg) | uint64_t(len);
}

template <bool kFiles>
__global__ void __launch_bounds__(kRowThreads) expand_root_kernel(const DevGrammar d, int64_t tiles,
                                                                  unsigned long long* __restrict__ look,
                                                                  const int4* __restrict__ ends,
                                                                  const int64_t* __restrict__ first, int file_bits,
                                                                  int32_t* __restrict__ words, int polls) {
  __shared__ int64_t s_warp[kRowThreads / 32];
  __shared__ int64_t s_item, s_prefix;
  __shared__ int32_t s_file[2];
  __shared__ int32_t s_words[kExpandWords];
  __shared__ uint16_t s_list[kRowTile];  // first words of the listed references
  __shared__ int s_staged, s_refs;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (tid == 0) {
    s_item = int64_t(atomicAdd(look + tiles, 1ull));
    s_staged = kExpandWords;
    s_refs = 0;
  }
  __syncthreads();
  const int64_t item = s_item, j0 = item * kRowTile + tid * kRowItems;
  int32_t sy[kRowItems];
  int64_t len = 0, ln[kRowItems];
#pragma unroll
  for (int k = 0; k < kRowItems; ++k) sy[k] = j0 + k < d.root_len ? d.sym[j0 + k] : -1;
#pragma unroll
  for (int k = 0; k < kRowItems; ++k) {
    ln[k] = sy[k] < 0 ? 0 : (sy[k] < d.V ? 1 : int64_t(d.exp_len[sy[k] - d.V]));
    len += ln[k];
  }
  int64_t incl = len;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int64_t u = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += u;
  }
  if (lane == 31) s_warp[warp] = incl;
  __syncthreads();
  int64_t before = incl - len, total = 0;
#pragma unroll
  for (int w = 0; w < kRowThreads / 32; ++w) {
    before += w < warp ? s_warp[w] : 0;
    total += s_warp[w];
  }
  if (tid == 0) publish_aggregate(look, item, uint64_t(total));
  int64_t o = before;
  if (ends) {
#pragma unroll
    for (int k = 0; k < kRowItems; ++k) {
      if (sy[k] >= d.V && ln[k] > 0 && ln[k] <= 4 && o + ln[k] <= kExpandWords) {
        const int4 e = ends[sy[k] - d.V];
        s_words[o] = e.x;
        if (ln[k] > 1) s_words[o + 1] = e.y;
        if (ln[k] == 4) s_words[o + 2] = e.z;
        if (ln[k] > 2) s_words[o + ln[k] - 1] = e.w;
      }
      o += ln[k];
    }
    o = before;
  }
#pragma unroll
  for (int k = 0; k < kRowItems; ++k) {
    const bool fits = sy[k] >= 0 && ln[k] > 0 && o + ln[k] <= kExpandWords;
    const bool ref = fits && sy[k] >= d.V && !(ends && ln[k] <= 4);
    if (ref || (fits && sy[k] < d.V)) s_words[o] = sy[k];
    const unsigned m = __ballot_sync(0xffffffffu, ref);
    int at = 0;
    if (lane == 0 && m) at = atomicAdd(&s_refs, __popc(m));
    at = __shfl_sync(0xffffffffu, at, 0);
    if (ref) s_list[at + __popc(m & ((1u << lane) - 1u))] = uint16_t(o);
    o += ln[k];
  }
  __syncthreads();
  for (int i = tid; i < s_refs; i += kRowThreads) {
    int q = s_list[i];
    walk_rule(d, s_words[q] - d.V, [&](int32_t w) { s_words[q++] = w; });
  }
  if (warp == 0) {
    __syncwarp();
    const int64_t p = warp_look_back(look, item, uint64_t(total), nullptr, polls, true,
                                     [&](int64_t t) { return expand_tile_flag(d.sym, d.exp_len, d.V, t); });
    if (lane == 0) s_prefix = p;
  }
  __syncthreads();
  const int64_t base = s_prefix;
  if (kFiles) {
    if (tid < 2 && total > 0)
      s_file[tid] = int32_t(upper_bound_dev(first, int64_t(d.F) + 1, tid ? base + total - 1 : base) - 1);
    __syncthreads();
  }
  if (total > kExpandWords) {  // the symbols from the first one on that does not fit
    o = before;
#pragma unroll
    for (int k = 0; k < kRowItems; ++k) {
      if (sy[k] >= 0 && o + ln[k] > kExpandWords) {
        if (o <= kExpandWords) s_staged = int(o);
        // a symbol's words are in one file
        const int32_t f = kFiles && ln[k] > 0 ? file_from(first, s_file[0], s_file[1], base + o) : 0;
        if (sy[k] < d.V) {
          words[base + o] = kFiles ? int32_t(uint32_t(sy[k]) << file_bits | uint32_t(f)) : sy[k];
        } else {
          int64_t q = base + o;
          walk_rule(d, sy[k] - d.V, [&](int32_t w) {
            words[q++] = kFiles ? int32_t(uint32_t(w) << file_bits | uint32_t(f)) : w;
          });
        }
      }
      o += ln[k];
    }
    __syncthreads();
  }
  const int staged = int(total < s_staged ? total : int64_t(s_staged));
  for (int i = tid; i < staged; i += kRowThreads) {
    const int32_t w = s_words[i];
    words[base + i] =
        kFiles ? int32_t(uint32_t(w) << file_bits | uint32_t(file_from(first, s_file[0], s_file[1], base + i))) : w;
  }
}

// cnt[f] = windows of file f (0 for f = F)
__global__ void file_windows_kernel(const uint64_t* __restrict__ file_len, int32_t F, int64_t* __restrict__ cnt) {
  for (int32_t f = blockIdx.x * blockDim.x + threadIdx.x; f <= F; f += gridDim.x * blockDim.x)
    cnt[f] = f < F && file_len[f] > 2 ? int64_t(file_len[f]) - 2 : 0;
}

// The file of every word.
__global__ void __launch_bounds__(kRowThreads) token_files_kernel(int64_t N, const int64_t* __restrict__ first, int32_t F,
                                                                  uint32_t* __restrict__ files) {
  __shared__ int32_t s_file[2];
  const int64_t p0 = int64_t(blockIdx.x) * kRowTile, p1 = min(N, p0 + kRowTile);
  if (threadIdx.x < 2) s_file[threadIdx.x] = int32_t(upper_bound_dev(first, int64_t(F) + 1, threadIdx.x ? p1 - 1 : p0) - 1);
  __syncthreads();
  for (int k = 0; k < kRowItems; ++k) {
    const int64_t p = p0 + k * kRowThreads + threadIdx.x;
    if (p < p1) files[p] = uint32_t(file_from(first, s_file[0], s_file[1], p));
  }
}

// Words of every file back to back (word << file_bits | file where that is not
// negative), and each file's first word (F + 1 offsets).
void expand_files(gt_grammar* g, Buf& words, Buf& first, cudaStream_t s, int file_bits = -1) {
  gt_ctx* ctx = g->ctx;
  const DevGrammar& d = g->d;
  const int64_t tiles = (d.root_len + kRowTile - 1) / kRowTile;
  words = Buf(ctx, size_t(d.N) * 4, s);
  first = Buf(ctx, size_t(d.F + 1) * 8, s);
  const bool by_ends = d.root_len >= kExpandEnds && d.R > 1;
  Buf ends(ctx, by_ends ? size_t(d.R) * 16 : 0, s);
  if (by_ends) run_rule_ends(g, ends.as<int4>(), s, true);
  Buf look(ctx, size_t(tiles + 1) * 8, s), len(ctx, size_t(d.F + 1) * 8, s), sc(ctx, scan_scratch_bytes(d.F + 1), s);
  file_len_i64_kernel<<<grid_for(int64_t(d.F) + 1, 256, ctx->num_sms * 8), 256, 0, s>>>(d.file_len, d.F,
                                                                                     len.as<int64_t>());
  GT_LAUNCH_CHECK();
  exclusive_scan_i64(len.as<int64_t>(), first.as<int64_t>(), d.F + 1, sc.p, s);
  if (tiles == 0) return;
  GT_CUDA(cudaMemsetAsync(look.p, 0, size_t(tiles + 1) * 8, s));
  (file_bits >= 0 ? expand_root_kernel<true> : expand_root_kernel<false>)<<<unsigned(tiles), kRowThreads, 0, s>>>(
      d, tiles, look.as<unsigned long long>(), by_ends ? ends.as<int4>() : nullptr, first.as<int64_t>(), file_bits,
      words.as<int32_t>(), look_back_polls());
  GT_LAUNCH_CHECK();
}

// One row (file, word, count) per distinct word of every file, *total of them: in
// (file, word) order, or in (word, file) order (by_word; the counts beside the
// words in pay, word << 32 | count).
struct WordRows {
  Buf word, file, cnt, total;
  Buf pay;
  bool by_word = false;
  int64_t bound = 0;
};

void bu_local_word_rows(gt_grammar* g, int kbw, cudaStream_t s, WordRows& out) {
  gt_ctx* ctx = g->ctx;
  const DevGrammar& d = g->d;
  const int64_t N = int64_t(d.N);
  const int cap = int(std::max<int64_t>(256, (g->max_file_len + 255) / 256 * 256));
  Phase ph(ctx, "bu_local", s);
  Buf soff(ctx, size_t(d.F + 1) * 8, s), flen(ctx, size_t(d.F + 1) * 8, s), sc(ctx, scan_scratch_bytes(d.F + 1), s);
  Buf sw(ctx, size_t(N) * 4, s), scn(ctx, size_t(N) * 4, s), nr(ctx, size_t(d.F + 1) * 8, s);
  Buf roff(ctx, size_t(d.F + 1) * 8, s);
  out.bound = N;
  out.word = Buf(ctx, size_t(N) * 4, s);
  out.file = Buf(ctx, size_t(N) * 4, s);
  out.cnt = Buf(ctx, size_t(N) * 8, s);
  out.total = Buf(ctx, 8, s);
  file_len_i64_kernel<<<grid_for(int64_t(d.F) + 1, 256, ctx->num_sms * 8), 256, 0, s>>>(d.file_len, d.F,
                                                                                     flen.as<int64_t>());
  GT_LAUNCH_CHECK();
  exclusive_scan_i64(flen.as<int64_t>(), soff.as<int64_t>(), d.F + 1, sc.p, s);
  const size_t smem = size_t(cap) * 8;
  GT_CUDA(cudaFuncSetAttribute(local_word_rows_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem)));
  GT_CUDA(cudaMemsetAsync(nr.as<int64_t>() + d.F, 0, 8, s));
  local_word_rows_kernel<<<unsigned(std::min<int64_t>(d.F, 65535)), kLocalThreads, smem, s>>>(
      d, cap, kbw, soff.as<int64_t>(), sw.as<int32_t>(), scn.as<uint32_t>(), nr.as<int64_t>());
  GT_LAUNCH_CHECK();
  exclusive_scan_i64(nr.as<int64_t>(), roff.as<int64_t>(), d.F + 1, sc.p, s);
  GT_CUDA(cudaMemcpyAsync(out.total.p, roff.as<int64_t>() + d.F, 8, cudaMemcpyDeviceToDevice, s));
  local_pack_kernel<<<grid_for(int64_t(d.F) * 32, 256, ctx->num_sms * 16), 256, 0, s>>>(
      d.F, soff.as<int64_t>(), roff.as<int64_t>(), sw.as<int32_t>(), scn.as<uint32_t>(), out.word.as<int32_t>(),
      out.file.as<int32_t>(), out.cnt.as<uint64_t>());
  GT_LAUNCH_CHECK();
}

void bu_word_rows(gt_grammar* g, cudaStream_t s, WordRows& out) {
  gt_ctx* ctx = g->ctx;
  const DevGrammar& d = g->d;
  const int threads = 256, cap = ctx->num_sms * 16;
  if (d.depth > kMaxStack) fail(GT_EOVERFLOW, "bottom-up expansion supports DAG depth <= 64");
  if (d.N >= (uint64_t(1) << 32)) fail(GT_EOVERFLOW, "per-file analytics need fewer than 2^32 tokens per grammar");
  const int kbw = bits_for(d.V);
  const int fb = bits_for(d.F);
  if (g->max_file_len <= kLocalMax && gparam(g, "bu_local", 1)) {
    bu_local_word_rows(g, kbw, s, out);
    return;
  }
  if (kbw + fb > 63) fail(GT_EOVERFLOW, "too many files x words for 64-bit (file, word) keys");
  // The expanded files come in file order, so a stable sort by word alone puts
  // their words in (word, file) order - the inverted index's - on 32-bit keys;
  // the distinct rows, about a third, then take two short passes to file order.
  // Rows of (file, word) keys take four passes, and the distinct ones three more
  // for the index.  Not if the expansion is far larger than the rows of the root
  // and its children.
  if (int64_t(d.N) <= 2 * (g->info.root_words + g->bu_words) && d.N < (uint64_t(1) << 30)) {
    Phase ph(ctx, "bu_rows", s);
    const int64_t N = int64_t(d.N);
    out.by_word = true;
    out.bound = N;
    out.word = Buf(ctx, size_t(N) * 4, s);
    out.file = Buf(ctx, size_t(N) * 4, s);
    out.pay = Buf(ctx, size_t(N) * 8, s);
    out.total = Buf(ctx, 8, s);
    if (N == 0) {
      GT_CUDA(cudaMemsetAsync(out.total.p, 0, 8, s));
      return;
    }
    Buf words, first, w1(ctx, size_t(N) * 4, s), rs(ctx, radix_scratch_bytes(N, true, 4), s);
    const int vbits = bits_for(std::max(d.V - 1, 1)), fbits = bits_for(std::max(d.F - 1, 1));
    RunOut o;
    o.pay = out.pay.as<uint64_t>();
    o.rows = out.total.as<int64_t>();
    if (vbits + fbits < 32) {
      // a row is one 32-bit word, sorted on its word bits: 8 bytes per row and pass
      // instead of 16 (2,000 files, 25M words: 1305 -> 1168 us)
      expand_files(g, words, first, s, fbits);
      const bool b = radix_sort_pingpong32(words.as<uint32_t>(), w1.as<uint32_t>(), nullptr, nullptr, 0, N, fbits,
                                           fbits + vbits, rs.p, s);
      o.low_bits = fbits;
      o.file = out.word.as<int32_t>();  // the high bits
      o.word = out.file.as<int32_t>();  // the low bits
      reduce_runs32(ctx, (b ? w1 : words).as<uint32_t>(), N, o, s);
      return;
    }
    Buf files(ctx, size_t(N) * 4, s), f1(ctx, size_t(N) * 4, s);
    expand_files(g, words, first, s);
    token_files_kernel<<<unsigned((N + kRowTile - 1) / kRowTile), kRowThreads, 0, s>>>(N, first.as<int64_t>(), d.F,
                                                                                      files.as<uint32_t>());
    GT_LAUNCH_CHECK();
    const bool b =
        radix_sort_pingpong32(words.as<uint32_t>(), w1.as<uint32_t>(), files.p, f1.p, 4, N, 0, vbits, rs.p, s);
    o.word = out.word.as<int32_t>();
    o.file = out.file.as<int32_t>();
    reduce_file_runs(ctx, (b ? w1 : words).as<uint32_t>(), (b ? f1 : files).as<uint32_t>(), N, nullptr, o, s);
    return;
  }
  const int64_t n = g->info.root_words + g->bu_words;
  Phase ph(ctx, "bu_rows", s);
  Buf k0(ctx, size_t(n) * 8, s), v0(ctx, size_t(n) * 4, s), k1(ctx, size_t(n) * 8, s), v1(ctx, size_t(n) * 4, s);
  Buf ecnt(ctx, size_t(d.ER) * 8, s), epos(ctx, size_t(d.ER) * 8, s), sc(ctx, scan_scratch_bytes(d.ER), s);
  Buf claimed(ctx, 8, s);
  if (g->info.root_words > 0) {
    GT_CUDA(cudaMemsetAsync(claimed.p, 0, 8, s));
    root_word_rows_kernel<<<unsigned((d.root_len + kRowTile - 1) / kRowTile), kRowThreads, 0, s>>>(
        d, kbw, claimed.as<unsigned long long>(), k0.as<uint64_t>(), v0.as<uint32_t>());
    GT_LAUNCH_CHECK();
  }
  if (d.ER > 0) {
    redge_len_kernel<<<grid_for(d.ER, threads, cap), threads, 0, s>>>(d, false, ecnt.as<int64_t>());
    GT_LAUNCH_CHECK();
    exclusive_scan_i64(ecnt.as<int64_t>(), epos.as<int64_t>(), d.ER, sc.p, s);
    child_word_rows_kernel<<<grid_for(d.ER, 128, cap), 128, 0, s>>>(d, kbw, epos.as<int64_t>(),
                                                                     k0.as<uint64_t>() + g->info.root_words,
                                                                     v0.as<uint32_t>() + g->info.root_words);
    GT_LAUNCH_CHECK();
  }
  out.bound = n;
  out.word = Buf(ctx, size_t(n) * 4, s);
  out.file = Buf(ctx, size_t(n) * 4, s);
  out.cnt = Buf(ctx, size_t(n) * 8, s);
  out.total = Buf(ctx, 8, s);
  if (n == 0) {
    GT_CUDA(cudaMemsetAsync(out.total.p, 0, 8, s));
    return;
  }
  Buf rs(ctx, radix_scratch_bytes(n, true, 4), s);
  const int kbits = kbw + bits_for(std::max(d.F - 1, 1));
  const bool b = radix_sort_pingpong(k0.as<uint64_t>(), k1.as<uint64_t>(), v0.p, v1.p, 4, n, 0, kbits, kbits, kbits,
                                     rs.p, s);
  RunOut o;
  o.low_bits = kbw;
  o.word = out.word.as<int32_t>();
  o.file = out.file.as<int32_t>();
  o.count = out.cnt.as<uint64_t>();
  o.rows = out.total.as<int64_t>();
  reduce_runs(ctx, (b ? k1 : k0).as<uint64_t>(), nullptr, (b ? v1 : v0).as<uint32_t>(), n, nullptr, ~uint64_t(0), o, s);
}

__global__ void unpack_pay_kernel(const uint64_t* __restrict__ pay, const int64_t* __restrict__ n_dev,
                                  int32_t* __restrict__ word, uint64_t* __restrict__ cnt) {
  const int64_t n = *n_dev;
  for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < n; i += int64_t(gridDim.x) * blockDim.x) {
    const uint64_t x = pay[i];
    if (word) word[i] = int32_t(x >> 32);
    cnt[i] = x & 0xffffffffu;
  }
}

// Rows in (word, file) order to (file, word) order: stable by file.
void rows_by_file(gt_grammar* g, WordRows& wr, cudaStream_t s) {
  if (!wr.by_word) return;
  gt_ctx* ctx = g->ctx;
  const int64_t n = wr.bound;
  const int64_t* nd = wr.total.as<int64_t>();
  wr.by_word = false;
  wr.cnt = Buf(ctx, size_t(n) * 8, s);
  if (n == 0) return;
  Buf f1(ctx, size_t(n) * 4, s), p1(ctx, size_t(n) * 8, s), rs(ctx, radix_scratch_bytes(n, true, 8), s);
  if (radix_sort_pingpong32(wr.file.as<uint32_t>(), f1.as<uint32_t>(), wr.pay.p, p1.p, 8, n, 0,
                            bits_for(std::max(g->d.F - 1, 1)), rs.p, s, nd)) {
    std::swap(wr.file, f1);
    std::swap(wr.pay, p1);
  }
  unpack_pay_kernel<<<grid_for(n, 256, ctx->num_sms * 16), 256, 0, s>>>(wr.pay.as<uint64_t>(), nd,
                                                                       wr.word.as<int32_t>(), wr.cnt.as<uint64_t>());
  GT_LAUNCH_CHECK();
}

__global__ void copy_files_kernel(const int32_t* __restrict__ file, const int64_t* __restrict__ n_dev,
                                  int32_t* __restrict__ out) {
  const int64_t n = *n_dev;
  for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < n; i += int64_t(gridDim.x) * blockDim.x)
    out[i] = file[i];
}

// off[w] = first row whose word is >= w
__global__ void word_starts_kernel(const int32_t* __restrict__ word, const int64_t* __restrict__ n_dev, int32_t V,
                                   int64_t* __restrict__ off) {
  const int64_t n = *n_dev;
  for (int64_t w = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; w <= V; w += int64_t(gridDim.x) * blockDim.x) {
    int64_t lo = 0, hi = n;
    while (lo < hi) {
      const int64_t mid = (lo + hi) >> 1;
      if (word[mid] < w) lo = mid + 1;
      else hi = mid;
    }
    off[w] = lo;
  }
}

gt_result* bu_inverted_index(gt_grammar* g, WordRows& wr, cudaStream_t s) {
  gt_ctx* ctx = g->ctx;
  const DevGrammar& d = g->d;
  const int threads = 256, cap = ctx->num_sms * 16;
  ResultBuilder rb(ctx, s);
  const int64_t n = wr.bound;
  const int64_t* nd = wr.total.as<int64_t>();
  auto* off = static_cast<int64_t*>(rb.alloc(size_t(d.V + 1) * 8));
  auto* files = static_cast<int32_t*>(rb.alloc(size_t(n) * 4));
  int64_t* len = rb.new_len_slot();
  GT_CUDA(cudaMemcpyAsync(len, nd, 8, cudaMemcpyDeviceToDevice, s));
  if (wr.by_word) {  // the rows are the postings
    word_starts_kernel<<<grid_for(int64_t(d.V) + 1, threads, cap), threads, 0, s>>>(wr.word.as<int32_t>(), nd, d.V, off);
    GT_LAUNCH_CHECK();
    copy_files_kernel<<<grid_for(n, threads, cap), threads, 0, s>>>(wr.file.as<int32_t>(), nd, files);
    GT_LAUNCH_CHECK();
    rb.field("offsets", off, int64_t(d.V) + 1);
    rb.field_dyn("file", files, len);
    return rb.finish();
  }
  Buf k0(ctx, size_t(n) * 8, s), k1(ctx, size_t(n) * 8, s), f0(ctx, size_t(n) * 4, s);
  if (n > 0) {
    Buf rs(ctx, radix_scratch_bytes(n, true, 4), s);
    const int bits = bits_for(std::max(d.V - 1, 1));
    // the sorted files have to land in the result: after an even number of
    // passes that is the buffer the rows start in
    const bool even = (bits + 7) / 8 % 2 == 0;
    uint32_t* fa = even ? reinterpret_cast<uint32_t*>(files) : f0.as<uint32_t>();
    uint32_t* fb = even ? f0.as<uint32_t>() : reinterpret_cast<uint32_t*>(files);
    word_keys_kernel<<<grid_for(n, threads, cap), threads, 0, s>>>(wr.word.as<int32_t>(), wr.file.as<int32_t>(), nd,
                                                                    k0.as<uint64_t>(), fa);
    GT_LAUNCH_CHECK();
    if (radix_sort_pingpong(k0.as<uint64_t>(), k1.as<uint64_t>(), fa, fb, 4, n, 0, bits, bits, bits, rs.p, s, nd) ==
        even)
      fail(GT_EINVAL, "unexpected number of sort passes");
    if (!even) std::swap(k0, k1);
  }
  word_offsets_kernel<<<grid_for(int64_t(d.V) + 1, threads, cap), threads, 0, s>>>(k0.as<uint64_t>(), nd, d.V, off);
  GT_LAUNCH_CHECK();
  rb.field("offsets", off, int64_t(d.V) + 1);
  rb.field_dyn("file", files, len);
  return rb.finish();
}

}  // namespace

// Term vectors from the rows (offsets from the file column), and the
// inverted index; one set of rows serves every query.
void run_file_batch_bu(gt_grammar* g, const int* tv_topk, int n_tv, gt_result** tv_out, gt_result** ii_out,
                       cudaStream_t s) {
  WordRows wr;
  bu_word_rows(g, s, wr);
  const DevGrammar& d = g->d;
  // rows in word order: the index first, the term vectors re-order them
  if (ii_out && wr.by_word) {
    *ii_out = bu_inverted_index(g, wr, s);
    ii_out = nullptr;
  }
  if (n_tv > 0) {
    rows_by_file(g, wr, s);
    Buf toff(g->ctx, size_t(d.F + 1) * 8, s);
    file_offsets_kernel<<<grid_for(int64_t(d.F) + 1, 256, 4096), 256, 0, s>>>(wr.file.as<int32_t>(),
                                                                              wr.total.as<int64_t>(), d.F,
                                                                              toff.as<int64_t>());
    GT_LAUNCH_CHECK();
    for (int i = 0; i < n_tv; ++i)
      tv_out[i] = tv_from_arrays(g->ctx, wr.word.as<int32_t>(), wr.cnt.as<uint64_t>(), toff.as<int64_t>(),
                                 wr.total.as<int64_t>(), wr.bound, d.F, tv_topk[i], uint64_t(g->max_file_len), s, d.V);
  }
  if (ii_out) *ii_out = bu_inverted_index(g, wr, s);
}

gt_result* run_ranked_words_bu(gt_grammar* g, cudaStream_t s) {
  WordRows wr;
  bu_word_rows(g, s, wr);
  const int64_t n = wr.bound;
  gt_ctx* ctx = g->ctx;
  Buf rkey(ctx, size_t(n) * 8, s);
  if (wr.by_word && g->d.F <= kMaxRankFiles) {  // rows in (key, file) order already
    wr.cnt = Buf(ctx, size_t(n) * 8, s);
    if (n > 0) {
      widen_i32_kernel<<<grid_for(n, 256, ctx->num_sms * 16), 256, 0, s>>>(
          wr.word.as<int32_t>(), wr.total.as<int64_t>(), rkey.as<uint64_t>());
      GT_LAUNCH_CHECK();
      unpack_pay_kernel<<<grid_for(n, 256, ctx->num_sms * 16), 256, 0, s>>>(
          wr.pay.as<uint64_t>(), wr.total.as<int64_t>(), nullptr, wr.cnt.as<uint64_t>());
      GT_LAUNCH_CHECK();
    }
    return ranked_from_key_rows(ctx, rkey, wr.file, wr.cnt, wr.total.as<int64_t>(), n, 0, g->d.F,
                                uint64_t(g->max_file_len), s);
  }
  rows_by_file(g, wr, s);
  if (n > 0) {
    widen_i32_kernel<<<grid_for(n, 256, ctx->num_sms * 16), 256, 0, s>>>(wr.word.as<int32_t>(), wr.total.as<int64_t>(),
                                                                          rkey.as<uint64_t>());
    GT_LAUNCH_CHECK();
  }
  return ranked_from_rows(ctx, rkey, wr.file, wr.cnt, wr.total.as<int64_t>(), n, 0, false, bits_for(g->d.V),
                          uint64_t(g->max_file_len), s);
}

// Per-file window rows of small files, built per file in shared memory.
void bu_local_window_rows(gt_grammar* g, int kb, cudaStream_t s, Windows& out) {
  gt_ctx* ctx = g->ctx;
  const DevGrammar& d = g->d;
  const int64_t N = int64_t(d.N);
  const int cap = int(std::max<int64_t>(256, (g->max_file_len + 255) / 256 * 256));
  Phase ph(ctx, "bu_local", s);
  Buf soff(ctx, size_t(d.F + 1) * 8, s), flen(ctx, size_t(d.F + 1) * 8, s), sc(ctx, scan_scratch_bytes(d.F + 1), s);
  Buf sk(ctx, size_t(N) * 8, s), scn(ctx, size_t(N) * 4, s), nr(ctx, size_t(d.F + 1) * 8, s);
  Buf roff(ctx, size_t(d.F + 1) * 8, s);
  out.n = N;
  out.reduced = true;
  out.keys = Buf(ctx, size_t(N) * 8, s);
  out.rfile = Buf(ctx, size_t(N) * 4, s);
  out.rcnt = Buf(ctx, size_t(N) * 8, s);
  out.total = Buf(ctx, 8, s);
  file_len_i64_kernel<<<grid_for(int64_t(d.F) + 1, 256, ctx->num_sms * 8), 256, 0, s>>>(d.file_len, d.F,
                                                                                     flen.as<int64_t>());
  GT_LAUNCH_CHECK();
  exclusive_scan_i64(flen.as<int64_t>(), soff.as<int64_t>(), d.F + 1, sc.p, s);
  const size_t smem = size_t(cap) * 16;
  GT_CUDA(cudaFuncSetAttribute(local_window_rows_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem)));
  GT_CUDA(cudaMemsetAsync(nr.as<int64_t>() + d.F, 0, 8, s));
  local_window_rows_kernel<<<unsigned(std::min<int64_t>(d.F, 65535)), kLocalThreads, smem, s>>>(
      d, cap, kb, 3 * kb, soff.as<int64_t>(), sk.as<uint64_t>(), scn.as<uint32_t>(), nr.as<int64_t>());
  GT_LAUNCH_CHECK();
  exclusive_scan_i64(nr.as<int64_t>(), roff.as<int64_t>(), d.F + 1, sc.p, s);
  GT_CUDA(cudaMemcpyAsync(out.total.p, roff.as<int64_t>() + d.F, 8, cudaMemcpyDeviceToDevice, s));
  local_pack_windows_kernel<<<grid_for(int64_t(d.F) * 32, 256, ctx->num_sms * 16), 256, 0, s>>>(
      d.F, soff.as<int64_t>(), roff.as<int64_t>(), sk.as<uint64_t>(), scn.as<uint32_t>(), out.keys.as<uint64_t>(),
      out.rfile.as<int32_t>(), out.rcnt.as<uint64_t>());
  GT_LAUNCH_CHECK();
}

// Per-file window rows: windows owned by the root in each file, plus every
// window inside each (file, root child) expansion, weighted by multiplicity.
void bu_window_rows(gt_grammar* g, Buf& ends, int kb, cudaStream_t s, Windows& out) {
  if (g->d.depth > kMaxStack) fail(GT_EOVERFLOW, "bottom-up expansion supports DAG depth <= 64");
  if (g->max_file_len <= kLocalMax && gparam(g, "bu_local", 1)) {
    bu_local_window_rows(g, kb, s, out);
    return;
  }
  FileRowBufs rows;
  const FileRows fr = rows.make(g->ctx, kb, g->d.F, bu_row_bound(g), s);
  bu_emit_windows(g, ends, kb, fr, s);
  sort_file_rows(g->ctx, rows, kb, g->d.F, s, out);
}

int64_t bu_row_bound(const gt_grammar* g) { return 2 * g->d.root_len + g->bu_windows; }

void bu_emit_windows(gt_grammar* g, Buf& ends, int kb, const FileRows& fr, cudaStream_t s) {
  gt_ctx* ctx = g->ctx;
  const DevGrammar& d = g->d;
  const int threads = 256, cap = ctx->num_sms * 16;
  if (d.depth > kMaxStack) fail(GT_EOVERFLOW, "bottom-up expansion supports DAG depth <= 64");
  Phase ph(ctx, "bu_rows", s);
  Buf ecnt(ctx, size_t(d.ER) * 8, s), epos(ctx, size_t(d.ER) * 8, s), sc(ctx, scan_scratch_bytes(d.ER), s);
  Buf first(ctx, 8, s);
  if (d.root_len > 0) {
    root_window_rows_kernel<<<unsigned((d.root_len + kTile - 1) / kTile), kRootWinThreads, 0, s>>>(d, ends.as<int4>(),
                                                                                                  kb, fr);
    GT_LAUNCH_CHECK();
  }
  if (d.ER > 0) {
    redge_len_kernel<<<grid_for(d.ER, threads, cap), threads, 0, s>>>(d, true, ecnt.as<int64_t>());
    GT_LAUNCH_CHECK();
    exclusive_scan_i64(ecnt.as<int64_t>(), epos.as<int64_t>(), d.ER, sc.p, s);
    GT_CUDA(cudaMemcpyAsync(first.p, fr.n, 8, cudaMemcpyDeviceToDevice, s));
    child_window_rows_kernel<<<grid_for(d.ER, 128, cap), 128, 0, s>>>(d, kb, epos.as<int64_t>(),
                                                                     first.as<unsigned long long>(), fr);
    GT_LAUNCH_CHECK();
    add_rows_kernel<<<1, 1, 0, s>>>(first.as<unsigned long long>(), g->bu_windows, fr.n);
    GT_LAUNCH_CHECK();
  }
}

namespace {

// One row per window, in text order: key and file.
__global__ void __launch_bounds__(kRowThreads) token_windows_kernel(const int32_t* __restrict__ words, int64_t N,
                                                                    const int64_t* __restrict__ first, int32_t F,
                                                                    const int64_t* __restrict__ row, int kb,
                                                                    uint64_t* __restrict__ keys,
                                                                    uint32_t* __restrict__ files) {
  __shared__ int32_t s_file[2];
  const int64_t p0 = int64_t(blockIdx.x) * kRowTile, p1 = min(N, p0 + kRowTile);
  if (threadIdx.x < 2) s_file[threadIdx.x] = int32_t(upper_bound_dev(first, int64_t(F) + 1, threadIdx.x ? p1 - 1 : p0) - 1);
  __syncthreads();
  const int32_t f_lo = s_file[0], f_hi = s_file[1];
#pragma unroll 4
  for (int k = 0; k < kRowItems; ++k) {
    const int64_t p = p0 + k * kRowThreads + threadIdx.x;
    if (p >= p1) continue;
    const int32_t lo = file_from(first, f_lo, f_hi, p);
    if (p + 2 >= first[lo + 1]) continue;
    const int64_t o = row[lo] + (p - first[lo]);
    keys[o] = pack_compact(words[p], words[p + 1], words[p + 2], kb);
    files[o] = uint32_t(lo);
  }
}

// ---- rank order inside the runs of a key --------------------------------------------

constexpr int kRankThread = 8;    // rows of a run put in order by one thread
constexpr int kRankWarp = 256;    // by one warp; longer runs by a CTA

// Files of a key: count descending, file ascending.  Most keys have one file.
__global__ void rank_short_kernel(const int64_t* __restrict__ off, const int64_t* __restrict__ nkeys,
                                  const int32_t* __restrict__ file, const uint64_t* __restrict__ cnt,
                                  int32_t* __restrict__ ofile, uint64_t* __restrict__ ocnt,
                                  unsigned long long* __restrict__ nlist, int64_t* __restrict__ mid,
                                  int64_t* __restrict__ lng) {
  const int64_t n = *nkeys;
  for (int64_t u = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; u < n; u += int64_t(gridDim.x) * blockDim.x) {
    const int64_t s = off[u], len = off[u + 1] - s;
    if (len == 1) {
      ofile[s] = file[s];
      ocnt[s] = cnt[s];
    } else if (len <= kRankThread) {
      for (int a = 0; a < int(len); ++a) {
        const uint64_t c = cnt[s + a];
        int r = 0;
        for (int b = 0; b < int(len); ++b) {
          const uint64_t x = cnt[s + b];
          r += x > c || (x == c && b < a);
        }
        ofile[s + r] = file[s + a];
        ocnt[s + r] = c;
      }
    } else if (len <= kRankWarp) {
      mid[atomicAdd(&nlist[0], 1ull)] = u;
    } else {
      lng[atomicAdd(&nlist[1], 1ull)] = u;
    }
  }
}

__global__ void rank_mid_kernel(const int64_t* __restrict__ off, const int32_t* __restrict__ file,
                                const uint64_t* __restrict__ cnt, int32_t* __restrict__ ofile,
                                uint64_t* __restrict__ ocnt, const unsigned long long* __restrict__ nlist,
                                const int64_t* __restrict__ mid) {
  const int lane = threadIdx.x & 31;
  const int64_t n = int64_t(nlist[0]), warps = (int64_t(gridDim.x) * blockDim.x) >> 5;
  for (int64_t q = (blockIdx.x * int64_t(blockDim.x) + threadIdx.x) >> 5; q < n; q += warps) {
    const int64_t s = off[mid[q]];
    const int len = int(off[mid[q] + 1] - s);
    for (int a = lane; a < len; a += 32) {
      const uint64_t c = cnt[s + a];
      int r = 0;
      for (int b = 0; b < len; ++b) {  // one address per step: a broadcast
        const uint64_t x = cnt[s + b];
        r += x > c || (x == c && b < a);
      }
      ofile[s + r] = file[s + a];
      ocnt[s + r] = c;
    }
  }
}

// Runs of up to kMaxRankFiles rows: a stable sort in shared memory by max_count -
// count, the row's place above it.
__global__ void __launch_bounds__(kLocalThreads) rank_long_kernel(
    const int64_t* __restrict__ off, const int32_t* __restrict__ file, const uint64_t* __restrict__ cnt,
    uint64_t max_count, int cbits, int cap, int32_t* __restrict__ ofile, uint64_t* __restrict__ ocnt,
    const unsigned long long* __restrict__ nlist, const int64_t* __restrict__ lng) {
  extern __shared__ __align__(16) uint32_t lsm[];
  uint64_t* ka = reinterpret_cast<uint64_t*>(lsm);
  uint64_t* kz = ka + cap;
  __shared__ uint32_t wcnt[kLocalWarps][256];
  __shared__ uint32_t dstart[256];
  __shared__ uint32_t dtot[kLocalWarps];
  const int64_t n = int64_t(nlist[1]);
  for (int64_t q = blockIdx.x; q < n; q += gridDim.x) {
    const int64_t s = off[lng[q]];
    const int len = int(off[lng[q] + 1] - s);
    for (int i = threadIdx.x; i < len; i += kLocalThreads)
      ka[i] = (uint64_t(i) << cbits) | (max_count - cnt[s + i]);
    __syncthreads();
    const uint64_t* r = local_sort(ka, kz, len, cbits, wcnt, dstart, dtot);
    for (int i = threadIdx.x; i < len; i += kLocalThreads) {
      ofile[s + i] = file[s + int64_t(r[i] >> cbits)];
      ocnt[s + i] = max_count - (r[i] & ((uint64_t(1) << cbits) - 1));
    }
    __syncthreads();
  }
}

}  // namespace

void bu_token_windows(gt_grammar* g, int kb, Buf& keys, Buf& files, Buf& n, cudaStream_t s) {
  gt_ctx* ctx = g->ctx;
  const DevGrammar& d = g->d;
  if (d.depth > kMaxStack) fail(GT_EOVERFLOW, "bottom-up expansion supports DAG depth <= 64");
  Phase ph(ctx, "bu_rows", s);
  const int64_t N = int64_t(d.N);
  keys = Buf(ctx, size_t(N) * 8, s);
  files = Buf(ctx, size_t(N) * 4, s);
  n = Buf(ctx, 8, s);
  Buf words, first, cnt(ctx, size_t(d.F + 1) * 8, s), row(ctx, size_t(d.F + 1) * 8, s);
  Buf sc(ctx, scan_scratch_bytes(d.F + 1), s);
  expand_files(g, words, first, s);
  file_windows_kernel<<<grid_for(int64_t(d.F) + 1, 256, ctx->num_sms * 8), 256, 0, s>>>(d.file_len, d.F,
                                                                                     cnt.as<int64_t>());
  GT_LAUNCH_CHECK();
  exclusive_scan_i64(cnt.as<int64_t>(), row.as<int64_t>(), d.F + 1, sc.p, s);
  GT_CUDA(cudaMemcpyAsync(n.p, row.as<int64_t>() + d.F, 8, cudaMemcpyDeviceToDevice, s));
  if (N == 0) return;
  token_windows_kernel<<<unsigned((N + kRowTile - 1) / kRowTile), kRowThreads, 0, s>>>(
      words.as<int32_t>(), N, first.as<int64_t>(), d.F, row.as<int64_t>(), kb, keys.as<uint64_t>(),
      files.as<uint32_t>());
  GT_LAUNCH_CHECK();
}

gt_result* ranked_from_key_rows(gt_ctx* ctx, Buf& rkey, Buf& rfile, Buf& rcnt, const int64_t* n_dev, int64_t bound,
                                int kb, int32_t F, uint64_t max_count, cudaStream_t s) {
  const int threads = 256, cap = ctx->num_sms * 16;
  ResultBuilder rb(ctx, s);
  Phase ph(ctx, "ranked", s);
  auto* off = static_cast<int64_t*>(rb.alloc(size_t(bound + 1) * 8));
  auto* okey = static_cast<uint64_t*>(rb.alloc(size_t(bound) * 8));
  auto* ofile = static_cast<int32_t*>(rb.alloc(size_t(bound) * 4));
  auto* ocnt = static_cast<uint64_t*>(rb.alloc(size_t(bound) * 8));
  int64_t* len_off = rb.new_len_slot();
  int64_t* len_key = rb.new_len_slot();
  int64_t* len_row = rb.new_len_slot();
  if (bound == 0) {
    GT_CUDA(cudaMemsetAsync(off, 0, 8, s));
    const int64_t one = 1;
    GT_CUDA(cudaMemcpyAsync(len_off, &one, 8, cudaMemcpyHostToDevice, s));
  } else {
    if (max_count >= (uint64_t(1) << 31)) fail(GT_EOVERFLOW, "ranked index counts need files below 2^31 tokens");
    GT_CUDA(cudaMemcpyAsync(len_row, n_dev, 8, cudaMemcpyDeviceToDevice, s));
    RunOut o;
    o.key = okey;
    o.kb = kb;
    o.off = off;
    o.off_end = n_dev;
    o.rows = len_key;
    o.rows1 = len_off;
    reduce_runs(ctx, rkey.as<uint64_t>(), nullptr, nullptr, bound, n_dev, ~uint64_t(0), o, s);
    const int64_t nm = bound / (kRankThread + 1) + 1, nl = bound / (kRankWarp + 1) + 1;
    Buf nlist(ctx, 16, s), mid(ctx, size_t(nm) * 8, s), lng(ctx, size_t(nl) * 8, s);
    GT_CUDA(cudaMemsetAsync(nlist.p, 0, 16, s));
    rank_short_kernel<<<grid_for(bound, threads, cap), threads, 0, s>>>(
        off, len_key, rfile.as<int32_t>(), rcnt.as<uint64_t>(), ofile, ocnt, nlist.as<unsigned long long>(),
        mid.as<int64_t>(), lng.as<int64_t>());
    GT_LAUNCH_CHECK();
    if (F > kRankThread) {
      rank_mid_kernel<<<grid_for(nm * 32, threads, ctx->num_sms * 8), threads, 0, s>>>(
          off, rfile.as<int32_t>(), rcnt.as<uint64_t>(), ofile, ocnt, nlist.as<unsigned long long>(),
          mid.as<int64_t>());
      GT_LAUNCH_CHECK();
    }
    if (F > kRankWarp) {
      int cbits = 1;
      while ((uint64_t(1) << cbits) <= max_count) ++cbits;
      const int room = (F + 255) / 256 * 256;  // a key's files
      const size_t smem = size_t(room) * 16;
      GT_CUDA(cudaFuncSetAttribute(rank_long_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem)));
      rank_long_kernel<<<unsigned(std::min<int64_t>(nl, 2 * ctx->num_sms)), kLocalThreads, smem, s>>>(
          off, rfile.as<int32_t>(), rcnt.as<uint64_t>(), max_count, cbits, room, ofile, ocnt,
          nlist.as<unsigned long long>(), lng.as<int64_t>());
      GT_LAUNCH_CHECK();
    }
  }
  rb.field_dyn("offsets", off, len_off);
  rb.field_dyn("key", okey, len_key);
  rb.field_dyn("file", ofile, len_row);
  rb.field_dyn("count", ocnt, len_row);
  return rb.finish();
}

}  // namespace gt
