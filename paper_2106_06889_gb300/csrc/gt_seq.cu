// Sequence count (l = 3) and the ranked inverted index (Section IV-C/D).
//
// Every 3-word window of a file lies inside the expansion of exactly one
// lowest rule occurrence: the rule whose body it crosses (it touches two or
// more body symbols).  That rule "owns" the window, and the window occurs as
// many times as the rule does (its top-down weight).  So instead of the
// paper's two traversal phases with retry-on-unready relaunches, the engine
//   1. builds the head/tail buffers bottom-up (first and last two words of
//      every rule's expansion);
//   2. enumerates, for every body position j, the windows that start in
//      symbol j and leave it: a word starts one window, a child rule with two
//      or more words starts two (at its last two words).  Their words come from
//      the symbol, the next two body symbols (look-ahead that stops at the end
//      of the rule, or of the file in the root) and children's head/tail
//      buffers - the boundary fix-up between rule pieces;
//   3. weights each window by its rule's weight (global counts) or by the
//      rule's per-file weights (per-file counts);
//   4. canonicalises: radix sort by key, then a segmented sum per key.
// For rule r this yields W_r + 2 S_r - 2 windows when all children expand to
// two or more words - Eq. 1's bound with l = 3, which is then exact.
#include <algorithm>

#include "gt_device.cuh"

namespace gt {
namespace {

// Exclusive prefix of v over the CTA (kWinThreads threads); *total gets the sum.
__device__ __forceinline__ int cta_excl_scan(int v, int* total) {
  __shared__ int warp_tot[kWinThreads / 32];
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
  for (int w = 0; w < kWinThreads / 32; ++w) {
    const int t = warp_tot[w];
    before += w < warp ? t : 0;
    all += t;
  }
  __syncthreads();
  *total = all;
  return before + incl - v;
}

// Global counts, compacted: every owned window gets one row, in body
// position order.  One CTA per tile of kTile symbols (4 per thread); each
// tile's first row comes from the per-grammar tile offsets (the windows of
// every tile counted and scanned once, seq_tile_offsets), and the emit pass
// ranks the windows inside the tile.
// Rows of rules nothing references (weight 0) get the pad key.  Rows past
// `bound` are not written; the status word records it.  A warp takes 128
// consecutive symbols, 32 at a time, so that two ballots give the rows' order;
// rows are staged in shared memory and written in one dense run per tile.
struct WinStage {
  uint64_t key[2 * kTile];
  uint32_t val[2 * kTile];
};

__global__ void __launch_bounds__(kWinThreads, 3) win_emit_kernel(DevGrammar d, const int4* __restrict__ ends,
                                                                  const uint64_t* __restrict__ wt, int kb,
                                                                  uint64_t key_pad,
                                                                  const int64_t* __restrict__ tile_off, int64_t bound,
                                                                  uint64_t* __restrict__ keys,
                                                                  uint32_t* __restrict__ vals,
                                                                  unsigned* __restrict__ status) {
  extern __shared__ __align__(16) unsigned char win_smem[];
  TileEnds& te = *reinterpret_cast<TileEnds*>(win_smem);
  WinStage& stage = *reinterpret_cast<WinStage*>(win_smem);  // takes the ends' room once they are read
  __shared__ int warp_tot[kWinThreads / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const unsigned lt = (1u << lane) - 1u;
  const int64_t t0 = int64_t(blockIdx.x) * kTile;
  const int64_t first = tile_off[blockIdx.x];
  load_tile_ends(d, ends, t0, te);
  uint64_t k[4][2];
  uint32_t w[4];
  int at[4], n = 0;  // at: the symbol's first row in the warp
  unsigned has = 0;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int i = warp * 128 + q * 32 + lane;
    const int64_t j = t0 + i;
    const int h = j < d.G ? windows_in(te, i, kb, k[q]) : 0;
    const unsigned b0 = __ballot_sync(0xffffffffu, h & 1), b1 = __ballot_sync(0xffffffffu, h & 2);
    has |= unsigned(h) << (2 * q);
    at[q] = n + __popc(b0 & lt) + __popc(b1 & lt);
    n += __popc(b0) + __popc(b1);
    w[q] = 0;
    if (h) w[q] = j < d.root_len ? uint32_t(wt[0]) : uint32_t(wt[d.sym_rule[j - d.first_rule_tile * kTile]]);
  }
  if (lane == 0) warp_tot[warp] = n;
  __syncthreads();  // also: the ends are read, the stage takes their room
  int before = 0, total = 0;
#pragma unroll
  for (int x = 0; x < kWinThreads / 32; ++x) {
    before += x < warp ? warp_tot[x] : 0;
    total += warp_tot[x];
  }
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    int o = before + at[q];
#pragma unroll
    for (int z = 0; z < 2; ++z)
      if ((has >> (2 * q + z)) & 1u) {
        stage.key[o] = w[q] ? k[q][z] : key_pad;
        stage.val[o] = w[q];
        ++o;
      }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < total; i += kWinThreads)
    if (first + i < bound) {
      keys[first + i] = stage.key[i];
      vals[first + i] = stage.val[i];
    }
  if (threadIdx.x == 0 && first + total > bound) atomicOr(status, ST_OVERFLOW);
}

// The same windows as rows of one word (key << kCodeBits | code): a window of
// weight 1 to 3 is one row, a heavier one a row per component of its weight.  The
// rows are sorted next, so their order is free: a tile claims its rows with one
// atomic; every window's first row goes through the stage, the others (none in the
// root's tiles) are written by their threads.  425 us for 41M symbols and 49M
// windows, like the (key, weight) form: bound by the latency of its phases, not by
// the 8 bytes per row it writes.
__global__ void __launch_bounds__(kWinThreads, 3) win_emit_coded_kernel(DevGrammar d, const int4* __restrict__ ends,
                                                                        const uint64_t* __restrict__ wt, int kb,
                                                                        unsigned long long* __restrict__ n_rows,
                                                                        int64_t bound, uint64_t* __restrict__ keys,
                                                                        unsigned* __restrict__ status) {
  extern __shared__ __align__(16) unsigned char win_smem[];
  TileEnds& te = *reinterpret_cast<TileEnds*>(win_smem);
  uint64_t* const stage = reinterpret_cast<uint64_t*>(win_smem);  // takes the ends' room once they are read
  __shared__ int warp_tot[kWinThreads / 32];
  __shared__ unsigned long long s_base;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const unsigned lt = (1u << lane) - 1u;
  const int64_t t0 = int64_t(blockIdx.x) * kTile;
  load_tile_ends(d, ends, t0, te);
  uint64_t k[4][2];
  uint32_t w[4];  // weight, then what the first row leaves of it
  int at[4], n = 0, more = 0;
  unsigned has = 0;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int i = warp * 128 + q * 32 + lane;
    const int64_t j = t0 + i;
    const int h = j < d.G ? windows_in(te, i, kb, k[q]) : 0;
    w[q] = 0;
    if (h) w[q] = j < d.root_len ? uint32_t(wt[0]) : uint32_t(wt[d.sym_rule[j - d.first_rule_tile * kTile]]);
    if (w[q]) has |= unsigned(h) << (2 * q);
  }
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const unsigned h = (has >> (2 * q)) & 3u;
    const unsigned b0 = __ballot_sync(0xffffffffu, h & 1u), b1 = __ballot_sync(0xffffffffu, h & 2u);
    at[q] = n + __popc(b0 & lt) + __popc(b1 & lt);
    n += __popc(b0) + __popc(b1);
    if (h) {
      const uint32_t code = take_code(w[q]);
      k[q][0] = k[q][0] << kCodeBits | code;
      k[q][1] = k[q][1] << kCodeBits | code;
      more += __popc(h) * int(weight_rows(w[q]));
    }
  }
  if (lane == 0) warp_tot[warp] = n;
  const int any_more = __syncthreads_or(more);  // also: the ends are read, the stage takes their room
  int before = 0, total = 0;
#pragma unroll
  for (int x = 0; x < kWinThreads / 32; ++x) {
    before += x < warp ? warp_tot[x] : 0;
    total += warp_tot[x];
  }
  int all_more = 0;
  int64_t my_more = any_more ? cta_excl_scan(more, &all_more) : 0;
  if (threadIdx.x == 0) s_base = total ? atomicAdd(n_rows, (unsigned long long)(total + all_more)) : 0ull;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    int o = before + at[q];
#pragma unroll
    for (int z = 0; z < 2; ++z)
      if ((has >> (2 * q + z)) & 1u) stage[o++] = k[q][z];
  }
  __syncthreads();
  const int64_t first = int64_t(s_base);
  if (first + total + all_more > bound) {  // cannot be: the bound holds for all weights
    if (threadIdx.x == 0) atomicOr(status, ST_OVERFLOW);
    return;
  }
  for (int i = threadIdx.x; i < total; i += kWinThreads) keys[first + i] = stage[i];
  if (more == 0) return;
  uint64_t* o = keys + first + total + my_more;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const unsigned h = (has >> (2 * q)) & 3u;
    if (!h) continue;
    while (w[q]) {
      const uint32_t code = take_code(w[q]);
#pragma unroll
      for (int z = 0; z < 2; ++z)
        if ((h >> z) & 1u) *o++ = (k[q][z] & ~uint64_t((1 << kCodeBits) - 1)) | code;
    }
  }
}

// Per-file rows, top-down: every window once per file of its rule (the root's
// once, in its own file), weighted by the rule's per-file weight.  A CTA counts
// the rows of its tile, claims their places with one atomic (the rows are
// sorted next, so their order is free) and writes them.  It replaced a count
// over all symbols, a scan of the counts and a second enumeration (61 + 40 + 79
// us on 7.1M symbols).
__global__ void __launch_bounds__(kWinThreads) win_emit_file_kernel(
    DevGrammar d, const int4* __restrict__ ends,
    const unsigned long long* __restrict__ mask, const int64_t* __restrict__ woff,
    const uint32_t* __restrict__ slot_pair, const uint32_t* __restrict__ fw, int kb, FileRows out) {
  __shared__ unsigned long long s_base;
  TileWin t;
  int32_t file[4];
  const int64_t j0 = int64_t(blockIdx.x) * kTile + threadIdx.x * 4;
  tile_windows(d, ends, kb, j0, t, file);
  unsigned long long m[4];
  int c = 0;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    m[i] = t.n[i] && t.r[i] ? mask[t.r[i]] : 0ull;
    c += t.n[i] * (t.r[i] ? __popcll(m[i]) : 1);
  }
  int total;
  const int before = cta_excl_scan(c, &total);
  if (threadIdx.x == 0) s_base = total ? atomicAdd(out.n, (unsigned long long)total) : 0ull;
  __syncthreads();
  int64_t o = int64_t(s_base) + before;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    if (t.n[i] == 0) continue;
    if (t.r[i] == 0) {
#pragma unroll
      for (int q = 0; q < 2; ++q)
        if (q < t.n[i]) out.put(o++, file[i], t.k[i][q], 1u);
    } else {
      int64_t slot = woff[t.r[i]];
      unsigned long long mm = m[i];
      while (mm) {
        const int f = __ffsll(mm) - 1;
        mm &= mm - 1;
        const uint32_t w = fw[slot_pair[slot++]];
#pragma unroll
        for (int q = 0; q < 2; ++q)
          if (q < t.n[i]) out.put(o++, f, t.k[i][q], w);
      }
    }
  }
}

__global__ void pad_tail_kernel(uint64_t* __restrict__ keys, uint32_t* __restrict__ vals,
                                const int64_t* __restrict__ n_dev, int64_t bound, uint64_t key_pad) {
  const int64_t n = *n_dev;
  for (int64_t i = n + blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < bound; i += int64_t(gridDim.x) * blockDim.x) {
    keys[i] = key_pad;
    vals[i] = 0;
  }
}

// Rows that are already one per (file, key): keys to 21-bit fields, copied.
__global__ void reduced_rows_out_kernel(const uint64_t* __restrict__ keys, const int32_t* __restrict__ file,
                                        const uint64_t* __restrict__ cnt, const int64_t* __restrict__ n_dev, int kb,
                                        uint64_t* __restrict__ okey, int32_t* __restrict__ ofile,
                                        uint64_t* __restrict__ ocnt) {
  const int64_t n = *n_dev;
  for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < n; i += int64_t(gridDim.x) * blockDim.x) {
    okey[i] = to_output_key(keys[i], kb);
    if (ofile) ofile[i] = file[i];
    ocnt[i] = cnt[i];
  }
}

int bits_for(int64_t x) {
  int b = 1;
  while ((int64_t(1) << b) <= x) ++b;
  return b;
}

}  // namespace

bool file_keys_fit(int kb, int32_t F) { return 3 * kb + bits_for(std::max(F - 1, 1)) < 64; }

// Buffers of the per-file window rows (at most `bound`; *n counts them).
FileRows FileRowBufs::make(gt_ctx* ctx, int kb, int32_t F, int64_t bound_, cudaStream_t s) {
  fits = file_keys_fit(kb, F);
  bound = bound_;
  keys = Buf(ctx, size_t(bound) * 8, s);
  vals = Buf(ctx, size_t(bound) * (fits ? 4 : 8), s);
  n = Buf(ctx, 8, s);
  GT_CUDA(cudaMemsetAsync(n.p, 0, 8, s));
  FileRows r;
  r.key = keys.as<uint64_t>();
  r.val = fits ? vals.as<uint32_t>() : nullptr;
  r.pay = fits ? nullptr : vals.as<uint64_t>();
  r.n = n.as<unsigned long long>();
  r.shift = 3 * kb;
  return r;
}

// Rows sorted by (file, key).  Where the file and the key fit one 64-bit word
// (file << 3 kb | key) that is one sort with 4-byte values: 24 bytes per row
// and pass.  Otherwise a stable sort by key carries (file << 32 | value) as a
// 64-bit payload and a second one, by the payload's file bits, carries the key:
// 32 bytes per row and pass.
void sort_file_rows(gt_ctx* ctx, FileRowBufs& r, int kb, int32_t F, cudaStream_t s, Windows& out) {
  out.n = r.bound;
  out.file_in_key = r.fits;
  if (r.bound == 0) return;
  Phase ph2(ctx, "seq_sort", s);
  const int64_t b = r.bound;
  const int vb = r.fits ? 4 : 8, fb = bits_for(std::max(F - 1, 1));
  const int64_t* nd = r.n.as<int64_t>();
  Buf k1(ctx, size_t(b) * 8, s), v1(ctx, size_t(b) * vb, s), rs(ctx, radix_scratch_bytes(b, true, vb), s);
  const int kbits = r.fits ? 3 * kb + fb : 3 * kb;
  if (radix_sort_pingpong(r.keys.as<uint64_t>(), k1.as<uint64_t>(), r.vals.p, v1.p, vb, b, 0, kbits, kbits, kbits, rs.p,
                          s, nd)) {
    std::swap(r.keys, k1);
    std::swap(r.vals, v1);
  }
  if (!r.fits && radix_sort_pingpong(r.vals.as<uint64_t>(), v1.as<uint64_t>(), r.keys.p, k1.p, 8, b, 32, 32 + fb,
                                     32 + fb, 32 + fb, rs.p, s, nd)) {
    std::swap(r.keys, k1);
    std::swap(r.vals, v1);
  }
  out.keys = std::move(r.keys);
  (r.fits ? out.vals : out.fkeys) = std::move(r.vals);
  out.n_dev = std::move(r.n);
}

namespace {

// Per-file window rows, top-down: windows x files of the rule.
int64_t td_row_bound(const gt_grammar* g) { return 2 * g->d.root_len + 2 * g->fsym_bound; }

void td_emit_windows(gt_grammar* g, Buf& ends, int kb, const FileRows& fr, cudaStream_t s) {
  const DevGrammar& d = g->d;
  Phase ph(g->ctx, "seq_emit", s);
  FileWeights fw;
  file_weights(g, s, fw);
  if (d.ntiles == 0) return;
  win_emit_file_kernel<<<unsigned(d.ntiles), kWinThreads, 0, s>>>(d, ends.as<int4>(), fw.mask, fw.off, fw.slot_pair,
                                                                 fw.w.as<uint32_t>(), kb, fr);
  GT_LAUNCH_CHECK();
}

// Device-detected failures of the global rows go to *status (the result's own status word).
void sorted_windows(gt_grammar* g, bool per_file, cudaStream_t s, Windows& out, uint32_t* status,
                    Buf* keep_ends = nullptr) {
  gt_ctx* ctx = g->ctx;
  const DevGrammar& d = g->d;
  const int threads = 256, cap = ctx->num_sms * 16;
  if (d.V > (1 << 21)) fail(GT_EOVERFLOW, "3-word keys need num_words <= 2^21");
  if (d.N >= (uint64_t(1) << 32)) fail(GT_EOVERFLOW, "sequence count needs fewer than 2^32 tokens per grammar");
  const int kb = bits_for(d.V > 1 ? d.V - 1 : 1);  // bits per word id
  out.kb = kb;
  // the pad sorts after every real key: all ones where that is none (word IDs below
  // 2^kb - 1 and so no bit of its own to sort on), else the next power of two
  const bool ones = d.V < (int64_t(1) << kb);
  out.key_pad = (uint64_t(1) << (3 * kb)) - (ones ? 1 : 0);
  const int key_bits = 3 * kb + (ones ? 0 : 1);
  Buf ends(ctx, size_t(d.R) * 16, s);
  {
    Phase ph(ctx, "seq_headtail", s);
    run_rule_ends(g, ends.as<int4>(), s, true);
  }
  const int64_t windows = g->info.owned_windows, tokens = int64_t(d.N);
  if (!per_file && windows > 0 && 3 * kb + kCodeBits <= 64 && tokens <= 3 * windows) {
    // Rows of one word, weight code and all: a pass moves 16 bytes per row instead
    // of 24.  The weights of the windows add up to the windows of all files, so a
    // row per component is at most windows + (tokens - windows) / 4 rows; three
    // tokens per window is where those rows take no more room than (key, weight)
    // rows.  100M nested words, 49M windows: the count and the word sort
    // take 3581 us so and 4131 us with (key, weight) rows.
    const int64_t bound = windows + std::max<int64_t>(tokens - windows, 0) / 4 + 1;
    Buf k0(ctx, size_t(bound) * 8, s), k1(ctx, size_t(bound) * 8, s);
    out.n_dev = Buf(ctx, 8, s);
    out.n = bound;
    out.max_runs = windows;
    out.coded = true;
    GT_CUDA(cudaMemsetAsync(out.n_dev.p, 0, 8, s));
    {
      Phase ph(ctx, "seq_emit", s);
      Buf wt(ctx, size_t(d.R) * 8, s);
      run_rule_weights(g, wt.as<uint64_t>(), s);
      constexpr size_t smem = std::max(sizeof(TileEnds), size_t(2 * kTile) * 8);
      GT_CUDA(cudaFuncSetAttribute(win_emit_coded_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem)));
      win_emit_coded_kernel<<<unsigned(d.ntiles), kWinThreads, smem, s>>>(
          d, ends.as<int4>(), wt.as<uint64_t>(), kb, out.n_dev.as<unsigned long long>(), bound, k0.as<uint64_t>(), status);
      GT_LAUNCH_CHECK();
    }
    Phase ph(ctx, "seq_sort", s);
    Buf rs(ctx, radix_scratch_bytes(bound, false, 0), s);
    const int hi = kCodeBits + 3 * kb;
    const bool b = radix_sort_pingpong(k0.as<uint64_t>(), k1.as<uint64_t>(), nullptr, nullptr, 0, bound, kCodeBits, hi,
                                       hi, hi, rs.p, s, out.n_dev.as<int64_t>());
    out.keys = std::move(b ? k1 : k0);
    if (keep_ends) *keep_ends = std::move(ends);
    return;
  }
  if (!per_file) {
    // exactly the owned windows (Eq. 1's count, known since load); the pad
    // key fills any rows the emit pass leaves
    const int64_t n = g->info.owned_windows;
    Buf k0(ctx, size_t(n) * 8, s), v0(ctx, size_t(n) * 4, s), k1(ctx, size_t(n) * 8, s), v1(ctx, size_t(n) * 4, s);
    out.n = n;
    if (n == 0) return;
    {
      Phase ph(ctx, "seq_emit", s);
      Buf wt(ctx, size_t(d.R) * 8, s);
      run_rule_weights(g, wt.as<uint64_t>(), s);
      const int64_t nt = d.ntiles;
      // each tile's first row: structure of the grammar, counted once and kept
      const int64_t* toff = seq_tile_offsets(g, ends.as<int4>(), kb, s);
      constexpr size_t smem = std::max(sizeof(TileEnds), sizeof(WinStage));
      GT_CUDA(cudaFuncSetAttribute(win_emit_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem)));
      win_emit_kernel<<<unsigned(nt), kWinThreads, smem, s>>>(d, ends.as<int4>(),
                                                            wt.as<uint64_t>(), kb, out.key_pad, toff, n,
                                                            k0.as<uint64_t>(), v0.as<uint32_t>(), status);
      GT_LAUNCH_CHECK();
      pad_tail_kernel<<<grid_for(n, threads, cap), threads, 0, s>>>(k0.as<uint64_t>(), v0.as<uint32_t>(), toff + nt, n,
                                                                     out.key_pad);
      GT_LAUNCH_CHECK();
    }
    Phase ph(ctx, "seq_sort", s);
    Buf rs(ctx, radix_scratch_bytes(n, true, 4), s);
    const bool b = radix_sort_pingpong(k0.as<uint64_t>(), k1.as<uint64_t>(), v0.p, v1.p, 4, n, 0, key_bits, key_bits,
                                       key_bits, rs.p, s);
    out.keys = std::move(b ? k1 : k0);
    out.vals = std::move(b ? v1 : v0);
    if (keep_ends) *keep_ends = std::move(ends);
    return;
  }
  if (file_strategy(g) == 2) {
    bu_window_rows(g, ends, kb, s, out);
    return;
  }
  FileRowBufs rows;
  const FileRows fr = rows.make(ctx, kb, d.F, td_row_bound(g), s);
  td_emit_windows(g, ends, kb, fr, s);
  sort_file_rows(ctx, rows, kb, d.F, s, out);
}

// One output row per distinct key of the sorted rows (per distinct (file, key)
// where they carry files); output_keys: keys with 21 bits per word.
void reduce_windows(gt_ctx* ctx, Windows& w, bool per_file, bool output_keys, uint64_t* key, int32_t* file,
                    uint64_t* count, int64_t* rows, cudaStream_t s) {
  RunOut o;
  o.key = key;
  o.kb = output_keys ? w.kb : 0;
  o.file = file;
  o.count = count;
  o.rows = rows;
  if (per_file && w.file_in_key) o.low_bits = 3 * w.kb;
  if (w.n == 0) {
    GT_CUDA(cudaMemsetAsync(rows, 0, 8, s));
    return;
  }
  if (w.coded) {
    reduce_coded_runs(ctx, w.keys.as<uint64_t>(), w.n, w.n_dev.as<int64_t>(), o, s);
    return;
  }
  // rows that carry files end at *n_dev and hold no pads
  reduce_runs(ctx, w.keys.as<uint64_t>(), per_file && !w.file_in_key ? w.fkeys.as<uint64_t>() : nullptr,
              w.vals.as<uint32_t>(), w.n, per_file ? w.n_dev.as<int64_t>() : nullptr,
              per_file ? ~uint64_t(0) : w.key_pad, o, s);
}

// (max_count - count) << 32 | file: ascending = count descending (counts of a
// key in a file never exceed max_count, the longest file's length).
__global__ void rank_keys_kernel(const uint64_t* __restrict__ cnt, const int32_t* __restrict__ file,
                                 const int64_t* __restrict__ n_dev, uint64_t max_count, uint64_t* __restrict__ k) {
  const int64_t n = *n_dev;
  for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < n; i += int64_t(gridDim.x) * blockDim.x)
    k[i] = ((max_count - cnt[i]) << 32) | uint32_t(file[i]);
}

// rkey[i] = key << cbits | (max_count - count), in place
__global__ void rank_key_count_kernel(const uint64_t* __restrict__ cnt, const int64_t* __restrict__ n_dev,
                                      uint64_t max_count, int cbits, uint64_t* __restrict__ rkey) {
  const int64_t n = *n_dev;
  for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < n; i += int64_t(gridDim.x) * blockDim.x)
    rkey[i] = (rkey[i] << cbits) | (max_count - cnt[i]);
}

// back to the key (in place), the count and the file
__global__ void rank_split_kernel(uint64_t* __restrict__ rkey, const int32_t* __restrict__ rfile,
                                  const int64_t* __restrict__ n_dev, uint64_t max_count, int cbits,
                                  int32_t* __restrict__ file, uint64_t* __restrict__ cnt) {
  const int64_t n = *n_dev;
  for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < n; i += int64_t(gridDim.x) * blockDim.x) {
    const uint64_t x = rkey[i];
    cnt[i] = max_count - (x & ((uint64_t(1) << cbits) - 1));
    rkey[i] = x >> cbits;
    file[i] = rfile[i];
  }
}

__global__ void rank_unpack_kernel(const uint64_t* __restrict__ pay, const int64_t* __restrict__ n_dev,
                                   uint64_t max_count, int32_t* __restrict__ file, uint64_t* __restrict__ cnt) {
  const int64_t n = *n_dev;
  for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < n; i += int64_t(gridDim.x) * blockDim.x) {
    const uint64_t x = pay[i];
    file[i] = int32_t(uint32_t(x));
    cnt[i] = max_count - (x >> 32);
  }
}

}  // namespace

// Rows (key, file, count), n_dev of them (bound allocated) -> ranked index:
// keys ascending; inside a key, count descending then file ascending.
gt_result* ranked_from_rows(gt_ctx* ctx, Buf& rkey, Buf& rfile, Buf& rcnt, const int64_t* n_dev, int64_t bound,
                            int kb, bool windows, int key_bits, uint64_t max_count, cudaStream_t s) {
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
  GT_CUDA(cudaMemcpyAsync(len_row, n_dev, 8, cudaMemcpyDeviceToDevice, s));
  if (bound == 0) {
    GT_CUDA(cudaMemsetAsync(off, 0, 8, s));
    GT_CUDA(cudaMemsetAsync(len_key, 0, 8, s));
    const int64_t one = 1;
    GT_CUDA(cudaMemcpyAsync(len_off, &one, 8, cudaMemcpyHostToDevice, s));
  } else {
    if (max_count >= (uint64_t(1) << 31)) fail(GT_EOVERFLOW, "ranked index counts need files below 2^31 tokens");
    const int cbits = bits_for(int64_t(max_count));  // max_count < 2^31
    Buf k1(ctx, size_t(bound) * 8, s), rs(ctx, radix_scratch_bytes(bound, true, 8), s);
    if (key_bits + cbits < 64) {
      // one sort by (key, max_count - count) carrying the file: stable, so the
      // files of equal counts stay ascending
      Buf f1(ctx, size_t(bound) * 4, s);
      rank_key_count_kernel<<<grid_for(bound, threads, cap), threads, 0, s>>>(rcnt.as<uint64_t>(), n_dev, max_count,
                                                                              cbits, rkey.as<uint64_t>());
      GT_LAUNCH_CHECK();
      const int bits = key_bits + cbits;
      if (radix_sort_pingpong(rkey.as<uint64_t>(), k1.as<uint64_t>(), rfile.p, f1.p, 4, bound, 0, bits, bits, bits, rs.p,
                              s, n_dev)) {
        std::swap(rkey, k1);
        std::swap(rfile, f1);
      }
      rank_split_kernel<<<grid_for(bound, threads, cap), threads, 0, s>>>(rkey.as<uint64_t>(), rfile.as<int32_t>(), n_dev,
                                                                          max_count, cbits, ofile, ocnt);
      GT_LAUNCH_CHECK();
    } else {
      // sort 1: stable by count descending, key ((max_count - count) << 32 |
      // file), payload the row key; sort 2: stable by row key, payload sort 1's key
      Buf k0(ctx, size_t(bound) * 8, s), v1(ctx, size_t(bound) * 8, s);
      rank_keys_kernel<<<grid_for(bound, threads, cap), threads, 0, s>>>(rcnt.as<uint64_t>(), rfile.as<int32_t>(), n_dev,
                                                                          max_count, k0.as<uint64_t>());
      GT_LAUNCH_CHECK();
      if (radix_sort_pingpong(k0.as<uint64_t>(), k1.as<uint64_t>(), rkey.p, v1.p, 8, bound, 32, 32 + cbits, 32 + cbits,
                              32 + cbits, rs.p, s, n_dev)) {
        std::swap(k0, k1);
        std::swap(rkey, v1);
      }
      if (radix_sort_pingpong(rkey.as<uint64_t>(), v1.as<uint64_t>(), k0.p, k1.p, 8, bound, 0, key_bits, key_bits,
                              key_bits, rs.p, s, n_dev)) {
        std::swap(k0, k1);
        std::swap(rkey, v1);
      }
      rank_unpack_kernel<<<grid_for(bound, threads, cap), threads, 0, s>>>(k0.as<uint64_t>(), n_dev, max_count, ofile,
                                                                            ocnt);
      GT_LAUNCH_CHECK();
    }
    RunOut o;
    o.key = okey;
    o.kb = windows ? kb : 0;
    o.off = off;
    o.off_end = n_dev;
    o.rows = len_key;
    o.rows1 = len_off;
    reduce_runs(ctx, rkey.as<uint64_t>(), nullptr, nullptr, bound, n_dev, ~uint64_t(0), o, s);
  }
  rb.field_dyn("offsets", off, len_off);
  rb.field_dyn("key", okey, len_key);
  rb.field_dyn("file", ofile, len_row);
  rb.field_dyn("count", ocnt, len_row);
  return rb.finish();
}

gt_result* reduce_key_rows(gt_ctx* ctx, Buf& keys, Buf& vals, int64_t n, int kb, int key_bits, cudaStream_t s,
                           const uint32_t* status_in, const int64_t* n_dev) {
  ResultBuilder rb(ctx, s);
  if (status_in) GT_CUDA(cudaMemcpyAsync(rb.status(), status_in, 4, cudaMemcpyDeviceToDevice, s));
  auto* key = static_cast<uint64_t*>(rb.alloc(size_t(n) * 8));
  auto* count = static_cast<uint64_t*>(rb.alloc(size_t(n) * 8));
  int64_t* len = rb.new_len_slot();
  if (n > 0) {
    Phase ph(ctx, "rows_sort", s);
    Buf k1(ctx, size_t(n) * 8, s), v1(ctx, size_t(n) * 4, s), rs(ctx, radix_scratch_bytes(n, true, 4), s);
    const bool b = radix_sort_pingpong(keys.as<uint64_t>(), k1.as<uint64_t>(), vals.p, v1.p, 4, n, 0, key_bits, key_bits,
                                       key_bits, rs.p, s, n_dev);
    RunOut o;
    o.key = key;
    o.kb = kb;
    o.count = count;
    o.rows = len;
    reduce_runs(ctx, (b ? k1 : keys).as<uint64_t>(), nullptr, (b ? v1 : vals).as<uint32_t>(), n, n_dev, ~uint64_t(0), o,
                s);
  } else {
    GT_CUDA(cudaMemsetAsync(len, 0, 8, s));
  }
  rb.field_dyn("key", key, len);
  rb.field_dyn("count", count, len);
  return rb.finish();
}

gt_result* run_ranked_windows(gt_grammar* g, cudaStream_t s) {
  gt_ctx* ctx = g->ctx;
  const DevGrammar& d = g->d;
  Windows w;
  // Rows sorted straight into (key, file) order, when a key has few enough files
  // to put in rank order afterwards: as one word (key << file bits | file), or,
  // if that is too wide, from the expanded files, whose windows come in file
  // order (not if the expansion is far larger than the rows of the root and its
  // children).  Sorting each file's windows first and then all rows by count and
  // by key takes two more sorts (8,000 short files: 1.9 against 1.1 ms of kernels).
  const int fb = bits_for(std::max(d.F - 1, 1)), kb = bits_for(std::max(d.V - 1, 1));
  const bool bottom_up = file_strategy(g) == 2, one_word = 3 * kb + fb < 64;
  if (d.F <= kMaxRankFiles && d.V <= (1 << 21) && d.N < (uint64_t(1) << 32) && (bottom_up || one_word) &&
      (one_word || int64_t(d.N) <= 2 * bu_row_bound(g))) {
    const int64_t bound = one_word ? (bottom_up ? bu_row_bound(g) : td_row_bound(g)) : int64_t(d.N);
    Buf rkey(ctx, size_t(bound) * 8, s), rfile(ctx, size_t(bound) * 4, s), rcnt(ctx, size_t(bound) * 8, s);
    Buf nd(ctx, 8, s);
    RunOut o;
    o.count = rcnt.as<uint64_t>();
    o.rows = nd.as<int64_t>();
    if (one_word) {
      Buf ends(ctx, size_t(d.R) * 16, s);
      {
        Phase ph(ctx, "seq_headtail", s);
        run_rule_ends(g, ends.as<int4>(), s, true);
      }
      FileRowBufs rows;
      FileRows fr = rows.make(ctx, kb, d.F, bound, s);
      fr.shift = 0;
      fr.key_shift = fb;
      if (bottom_up) bu_emit_windows(g, ends, kb, fr, s);
      else td_emit_windows(g, ends, kb, fr, s);
      if (bound > 0) {
        Buf k1(ctx, size_t(bound) * 8, s), v1(ctx, size_t(bound) * 4, s), rs(ctx, radix_scratch_bytes(bound, true, 4), s);
        const bool b = radix_sort_pingpong(rows.keys.as<uint64_t>(), k1.as<uint64_t>(), rows.vals.p, v1.p, 4, bound, 0,
                                           3 * kb + fb, 3 * kb + fb, 3 * kb + fb, rs.p, s, rows.n.as<int64_t>());
        o.low_bits = fb;
        o.hi = rkey.as<uint64_t>();
        o.word = rfile.as<int32_t>();
        reduce_runs(ctx, (b ? k1 : rows.keys).as<uint64_t>(), nullptr, (b ? v1 : rows.vals).as<uint32_t>(), bound,
                    rows.n.as<int64_t>(), ~uint64_t(0), o, s);
      }
    } else {
      Buf keys, files, n;
      bu_token_windows(g, kb, keys, files, n, s);
      if (bound > 0) {
        Buf k1(ctx, size_t(bound) * 8, s), f1(ctx, size_t(bound) * 4, s), rs(ctx, radix_scratch_bytes(bound, true, 4), s);
        const bool b = radix_sort_pingpong(keys.as<uint64_t>(), k1.as<uint64_t>(), files.p, f1.p, 4, bound, 0, 3 * kb,
                                           3 * kb, 3 * kb, rs.p, s, n.as<int64_t>());
        o.key = rkey.as<uint64_t>();
        o.file = rfile.as<int32_t>();
        reduce_file_runs(ctx, (b ? k1 : keys).as<uint64_t>(), (b ? f1 : files).as<uint32_t>(), bound, n.as<int64_t>(), o,
                         s);
      }
    }
    return ranked_from_key_rows(ctx, rkey, rfile, rcnt, nd.as<int64_t>(), bound, kb, d.F, uint64_t(g->max_file_len), s);
  }
  sorted_windows(g, true, s, w, nullptr);
  if (w.reduced)
    return ranked_from_rows(ctx, w.keys, w.rfile, w.rcnt, w.total.as<int64_t>(), w.n, w.kb, true, 3 * w.kb,
                            uint64_t(g->max_file_len), s);
  // per-file 3-gram rows (file, key, count) in (file, key) order
  Buf rkey(ctx, size_t(w.n) * 8, s), rfile(ctx, size_t(w.n) * 4, s), rcnt(ctx, size_t(w.n) * 8, s), nd(ctx, 8, s);
  reduce_windows(ctx, w, true, false, rkey.as<uint64_t>(), rfile.as<int32_t>(), rcnt.as<uint64_t>(), nd.as<int64_t>(),
                 s);
  return ranked_from_rows(ctx, rkey, rfile, rcnt, nd.as<int64_t>(), w.n, w.kb, true, 3 * w.kb,
                          uint64_t(g->max_file_len), s);
}

gt_result* run_sequence_count(gt_grammar* g, int per_file, cudaStream_t s, Buf* keep_ends) {
  // global count: the one-row-per-window radix sort (default, measured faster
  // on the 500M-token corpus) or the sample-sort buckets (seq_path = 2)
  if (!per_file && gparam(g, "seq_path", 1) == 2) return run_sequence_count_global(g, s);
  gt_ctx* ctx = g->ctx;
  ResultBuilder rb(ctx, s);
  Windows w;
  sorted_windows(g, per_file != 0, s, w, rb.status(), keep_ends);
  Phase ph(ctx, "seq_reduce", s);
  const int64_t runs = w.coded ? w.max_runs : w.n;
  auto* key = static_cast<uint64_t*>(rb.alloc(size_t(runs) * 8));
  auto* count = static_cast<uint64_t*>(rb.alloc(size_t(runs) * 8));
  int32_t* file = per_file ? static_cast<int32_t*>(rb.alloc(size_t(w.n) * 4)) : nullptr;
  int64_t* len = rb.new_len_slot();
  if (w.reduced) {
    GT_CUDA(cudaMemcpyAsync(len, w.total.p, 8, cudaMemcpyDeviceToDevice, s));
    if (w.n > 0) {
      reduced_rows_out_kernel<<<grid_for(w.n, 256, ctx->num_sms * 16), 256, 0, s>>>(
          w.keys.as<uint64_t>(), w.rfile.as<int32_t>(), w.rcnt.as<uint64_t>(), w.total.as<int64_t>(), w.kb, key, file,
          count);
      GT_LAUNCH_CHECK();
    }
  } else {
    reduce_windows(ctx, w, per_file != 0, true, key, file, count, len, s);
  }
  if (per_file) rb.field_dyn("file", file, len);
  rb.field_dyn("key", key, len);
  rb.field_dyn("count", count, len);
  return rb.finish();
}

}  // namespace gt
