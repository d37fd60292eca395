// Device helpers shared by the kernels: a search routine and the 3-word
// window helpers used by the global and per-file sequence paths.
#pragma once

#include <cstdint>
#include <type_traits>

#include "gt_internal.cuh"

namespace gt {

// ---- rows of one word: key << kCodeBits | code of a weight -----------------------
// A code stands for m x 4^s (m 1 to 3 in its low bits, s above), or for 2^8, 2^12,
// 2^16, 2^20 (m 0).  A weight takes one row per component: 1 to 3 take one, and a
// weight w at most 1 + (w - 1) / 4.
constexpr int kCodeBits = 4;

__device__ __forceinline__ uint32_t code_weight(uint32_t code) {
  const uint32_t m = code & 3u, s = (code >> 2) & 3u;
  return m ? m << (2 * s) : 256u << (4 * s);
}

// rows that a weight takes
__device__ __forceinline__ uint32_t weight_rows(uint32_t w) {
  return uint32_t(__popc((w | (w >> 1)) & 0x55u)) + ((w >> 8) & 15u) + ((w >> 12) & 15u) + ((w >> 16) & 15u) + (w >> 20);
}

// code of a component of w > 0, and what is left of w without it
__device__ __forceinline__ uint32_t take_code(uint32_t& w) {
  if (w & 0xffu) {
    const uint32_t s = uint32_t(__ffs(int(w & 0xffu)) - 1) >> 1, m = (w >> (2 * s)) & 3u;
    w &= ~(3u << (2 * s));
    return s << 2 | m;
  }
  const uint32_t s = (w & 0xf00u) ? 0u : (w & 0xf000u) ? 1u : (w & 0xf0000u) ? 2u : 3u;
  w -= 256u << (4 * s);
  return s << 2;
}

// Lanes of the warp holding the same 8-bit digit as this lane (among `active`),
// from one ballot per digit bit.  Every lane of the warp must call it.  Bound by
// instruction issue in the sort that ranks 32 rows per call: the bit's predicate
// both votes and selects a mask, ready with the ballot, that turns the ballot into
// the lanes that agree with this one.
__device__ __forceinline__ unsigned digit_bit_peers(uint32_t d, int b, unsigned peers) {
  asm volatile(
      "{\n\t"
      ".reg .pred has;\n\t"
      ".reg .b32 flip, votes;\n\t"
      "and.b32 flip, %1, %2;\n\t"
      "setp.ne.b32 has, flip, 0;\n\t"
      "selp.b32 flip, 0, -1, has;\n\t"
      "vote.sync.ballot.b32 votes, has, 0xffffffff;\n\t"
      "lop3.b32 %0, %0, votes, flip, 0x60;\n\t"  // peers and (votes xor flip)
      "}"
      : "+r"(peers)
      : "r"(d), "r"(1 << b));
  return peers;
}

// mask (uniform): the digit's bits; the ballots of bits 6 and 7 are skipped where it has none.
__device__ __forceinline__ unsigned warp_digit_peers(uint32_t d, unsigned active, uint32_t mask = 0xffu) {
  unsigned peers = active;
#pragma unroll
  for (int b = 0; b < 6; ++b) peers = digit_bit_peers(d, b, peers);
  if (mask & 0xc0u) {
    peers = digit_bit_peers(d, 6, peers);
    if (mask & 0x80u) peers = digit_bit_peers(d, 7, peers);
  }
  return peers;
}

// ---- chains of small DAG levels in one launch -----------------------------
// A level pass over a few thousand items is all latency: a launch, dependent
// loads, and the next level's launch.  The small levels of a grammar (kTailItems
// items at most, two per thread) run instead inside one thread-block cluster,
// whose hardware barrier separates the levels (release / acquire at cluster
// scope orders the global writes too; values written by earlier levels are read
// through L2).  A level's structure is requested before the barrier that its
// values wait for.  What it saves is the host's time per launch, about 4.5 us: 11
// levels launched one by one / in one cluster, us, by the items of a level:
//   weights    500: 55 / 28   4k: 56 / 29   8k: 56 / 29   12k: 56 / 34   16k: 56 / 36
//   ends       500: 59 / 35   4k: 59 / 38   8k: 59 / 39   12k: 59 / 53   16k: 59 / 54
//   per file   500: 114 / 86  4k: 124 / 103 8k: 130 / 108 12k: 130 / 110 16k: 130 / 110
// (with the rest of a head/tail call and of a term vector).  In a replayed graph a
// launch costs less than the barrier, and the levels keep theirs while a stream is
// captured: a word count by a plan 500: 43.5 / 45.7, 8k: 48 / 50, 16k: 52 / 59, a
// term vector 1k: 54 / 61, 4k: 64 / 74, a 3-word count 12k: 93 / 112.  Levels of more
// than kTailItems need more than a cluster's threads.
constexpr int kTailCtas = 8, kTailThreads = 1024;
constexpr int64_t kTailItems = 2 * kTailCtas * kTailThreads;

__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

__device__ __forceinline__ int64_t upper_bound_dev(const int64_t* a, int64_t n, int64_t x) {
  int64_t lo = 0, hi = n;
  while (lo < hi) {
    int64_t mid = (lo + hi) >> 1;
    if (a[mid] <= x) lo = mid + 1;
    else hi = mid;
  }
  return lo;
}

// ---- 3-word windows (shared by the top-down and bottom-up sequence paths) ----

struct Sym3 {
  int32_t first, second, second_last, last;  // -1 where the expansion is too short
};

__device__ __forceinline__ Sym3 sym_words(const DevGrammar& d, const int4* __restrict__ ends, int32_t x) {
  Sym3 r;
  if (x < d.V) {
    r.first = r.last = x;
    r.second = r.second_last = -1;
  } else {
    const int32_t c = x - d.V;
    const int4 e = ends[c];
    r = {e.x, e.y, e.z, e.w};
  }
  return r;
}

__device__ __forceinline__ uint64_t pack_compact(int32_t a, int32_t b, int32_t c, int kb) {
  return (uint64_t(uint32_t(a)) << (2 * kb)) | (uint64_t(uint32_t(b)) << kb) | uint64_t(uint32_t(c));
}

// End (exclusive) of the body sequence holding position j: the file's end in
// the root, the rule's end elsewhere.  Also returns the rule.
__device__ __forceinline__ int64_t seq_end(const DevGrammar& d, int64_t j, int32_t* rule, int32_t* file) {
  if (j < d.root_len) {
    const int64_t f = upper_bound_dev(d.file_off, int64_t(d.F) + 1, j) - 1;
    *rule = 0;
    *file = int32_t(f);
    return d.file_off[f + 1];
  }
  const int32_t r = d.sym_rule[j - d.first_rule_tile * kTile];
  *rule = r;
  *file = -1;
  return d.rule_off[r + 1];
}

// The (at most two) owned windows starting in body symbol j; returns how many.
__device__ __forceinline__ int windows_at(const DevGrammar& d, const int4* __restrict__ ends, int64_t j, int64_t end, int kb,
                                          uint64_t* k) {
  if (j + 1 >= end) return 0;
  const Sym3 a = sym_words(d, ends, d.sym[j]);
  const Sym3 b = sym_words(d, ends, d.sym[j + 1]);
  const int32_t n1 = b.first;
  int32_t n2 = b.second;
  if (n2 < 0) n2 = j + 2 < end ? sym_words(d, ends, d.sym[j + 2]).first : -1;
  // k[0], k[1] are always written (fixed indices keep them in registers)
  const bool w0 = a.second_last >= 0;  // child with >= 2 words
  const uint64_t x0 = w0 ? pack_compact(a.second_last, a.last, n1, kb) : 0;
  const uint64_t x1 = n2 >= 0 ? pack_compact(a.last, n1, n2, kb) : 0;
  k[0] = w0 ? x0 : x1;
  k[1] = x1;
  return int(w0) + int(n2 >= 0);
}

// Windows of the 4 symbols j0 .. j0+3: symbol i has n[i] of them, keys
// k[i][0..n[i]), owner rule r[i].
struct TileWin {
  uint64_t k[4][2];
  int32_t r[4];
  int n[4];
};

// file (optional): the file of each symbol of the root.
__device__ __forceinline__ int tile_windows(const DevGrammar& d, const int4* __restrict__ ends, int kb, int64_t j0, TileWin& t,
                                            int32_t* file = nullptr) {
  int c = 0;
  int64_t end = -1;  // end of the body sequence holding the previous symbol (rule or root file)
  int32_t rule = 0, f = -1;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int64_t j = j0 + i;
    t.n[i] = 0;
    t.r[i] = 0;
    if (j < d.G) {
      // the four symbols usually share one sequence: look it up again only
      // when the previous one ended (or at a root / rule boundary)
      if (j >= end || j == d.root_len) end = seq_end(d, j, &rule, &f);
      t.r[i] = rule;
      if (file) file[i] = f;
      t.n[i] = windows_at(d, ends, j, end, kb, t.k[i]);
    }
    c += t.n[i];
  }
  return c;
}

// ---- windows of a tile from shared memory -----------------------------------
// The words at both ends of every symbol of a tile (and of the two after it),
// looked up once per symbol, and a bit per symbol that ends its body sequence
// (file or rule).  A symbol's windows then need only its neighbours' entries:
// enumerating them from global memory looked up each symbol's ends three times,
// in dependent loads (with the rows staged too: 502 -> 423 us for 49M windows).
constexpr int kWinThreads = kTile / 4;

struct TileEnds {
  int4 words[kTile + 2];  // first, second, second to last, last (-1 where there is none)
  uint32_t last[kTile / 32 + 1];
};

// By the whole CTA (kWinThreads threads).
__device__ __forceinline__ void load_tile_ends(const DevGrammar& d, const int4* __restrict__ ends, int64_t t0, TileEnds& e) {
  const int tid = threadIdx.x;
  if (tid <= kTile / 32) e.last[tid] = 0;
  __syncthreads();
#pragma unroll
  for (int q = 0; q < 5; ++q) {
    const int i = q * kWinThreads + tid;
    if (i >= kTile + 2) break;
    const int64_t j = t0 + i;
    int4 w = make_int4(-1, -1, -1, -1);
    if (j < d.G) {
      const int32_t s = d.sym[j];
      if (s < d.V) {
        w.x = w.w = s;
      } else {
        w = ends[s - d.V];
      }
      if (j >= d.root_len && i <= kTile) {
        const int32_t* sr = d.sym_rule + (j - d.first_rule_tile * kTile);
        if (j + 1 == d.G || sr[0] != sr[1]) atomicOr(&e.last[i >> 5], 1u << (i & 31));
      }
    }
    e.words[i] = w;
  }
  if (t0 < d.root_len) {  // files that end in the tile (an empty one marks the end before it again)
    const int64_t t1 = t0 + kTile + 1;
    const int64_t f0 = upper_bound_dev(d.file_off, int64_t(d.F) + 1, t0);  // first f with file_off[f] > t0
    for (int64_t f = f0 + tid; f <= d.F; f += kWinThreads) {
      const int64_t i = d.file_off[f] - 1 - t0;
      if (d.file_off[f] > t1) break;
      atomicOr(&e.last[i >> 5], 1u << (i & 31));
    }
  }
  __syncthreads();
}

// The windows starting in symbol i of the tile, in text order: bit 0 of the
// result says that k[0] is one (a child of two or more words), bit 1 that k[1] is.
__device__ __forceinline__ int windows_in(const TileEnds& e, int i, int kb, uint64_t* k) {
  if ((e.last[i >> 5] >> (i & 31)) & 1u) return 0;
  const int4 a = e.words[i], b = e.words[i + 1];
  int32_t n2 = b.y;
  if (n2 < 0 && !((e.last[(i + 1) >> 5] >> ((i + 1) & 31)) & 1u)) n2 = e.words[i + 2].x;
  const bool w0 = a.z >= 0, w1 = n2 >= 0;
  k[0] = w0 ? pack_compact(a.z, a.w, b.x, kb) : 0;
  k[1] = w1 ? pack_compact(a.w, b.x, n2, kb) : 0;
  return int(w0) | int(w1) << 1;
}

// compact key (kb bits per word) -> w1 << 42 | w2 << 21 | w3; kb == 0 keeps it
__device__ __forceinline__ uint64_t to_output_key(uint64_t k, int kb) {
  if (kb == 0) return k;
  const uint64_t m = (uint64_t(1) << kb) - 1;
  return ((k >> (2 * kb)) << 42) | (((k >> kb) & m) << 21) | (k & m);
}

// ---- decoupled look-back over items taken in ticket order --------------
// Flag word per item: state in the top two bits (0 nothing published, 1 the
// item's own total, 2 the inclusive prefix through the item), value below.
// An item only waits on items with smaller tickets, i.e. ones already
// running, so every wait ends; each is bounded anyway.  What follows a wait
// that ran out depends on the caller: the primitives (scan, radix sort, run
// reduction, root expansion) work the missing item's value out of its input
// themselves and go on - a later kernel takes their output for indices, and the
// grammar keeps some of it, so it has to be right whatever happened - and the
// inverted index and the bucket path, whose output goes to the caller only,
// record ST_TIMEOUT.
constexpr uint64_t kFlagAgg = 1ull << 62, kFlagIncl = 2ull << 62, kFlagVal = (1ull << 62) - 1;
constexpr int kSpinLimit = 1 << 22;  // look-back polls before giving up (>= 0.25 s)

__device__ __forceinline__ unsigned long long ld_acquire_u64(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}

// The item's own total, published as soon as it is known (one thread); item
// 0 publishes its inclusive prefix directly.
__device__ __forceinline__ void publish_aggregate(unsigned long long* flags, int64_t item, uint64_t agg) {
  atomicExch(&flags[item], (item == 0 ? kFlagIncl : kFlagAgg) | agg);
}

struct NoRedo {};

// By one warp: reads the flags of the 32 preceding items at once, adds their
// values up to the nearest one with a published prefix, and moves 32 items
// further back while there is none; then publishes the item's inclusive
// prefix.  Returns the exclusive prefix (to every lane).  After spin_limit polls
// in which an item published nothing, redo(item) (called by the whole warp)
// gives the flag word it would have published; without redo it sets ST_TIMEOUT
// in *status, still publishes (so that later items are not held up) and returns
// -1.  publish == false: the item's own word already holds its final value.
template <class Redo = NoRedo>
__device__ __forceinline__ int64_t warp_look_back(unsigned long long* flags, int64_t item, uint64_t agg,
                                                  unsigned* status, int spin_limit = kSpinLimit, bool publish = true,
                                                  Redo redo = Redo()) {
  const int lane = threadIdx.x & 31;
  if (item == 0) return 0;
  uint64_t excl = 0;
  int64_t top = item - 1;  // the window is flags[top - 31 .. top], lane l reads top - l
  int spins = 0;
  bool ok = true;
  while (true) {
    const int64_t j = top - lane;
    unsigned long long v = j >= 0 ? ld_acquire_u64(&flags[j]) : kFlagIncl;
    uint64_t st = v & ~kFlagVal;
    if (__any_sync(0xffffffffu, st == 0)) {
      if (++spins <= spin_limit) {
        __nanosleep(32);
        continue;
      }
      if constexpr (std::is_same<Redo, NoRedo>::value) {
        ok = false;
        break;
      } else {  // the missing items before the nearest prefix, one after the other
#pragma unroll 1
        for (int l = 0; l < 32; ++l) {
          const uint64_t seen = __shfl_sync(0xffffffffu, st, l);
          if (seen == kFlagIncl) break;
          if (seen) continue;
          const uint64_t x = redo(top - l);
          if (lane == l) {
            v = x;
            st = x & ~kFlagVal;
          }
          if ((x & ~kFlagVal) == kFlagIncl) break;
        }
      }
    }
    const unsigned incl = __ballot_sync(0xffffffffu, st == kFlagIncl);
    const int stop = incl ? __ffs(incl) - 1 : 31;  // nearest item with a prefix, else the whole window
    uint64_t part = lane <= stop ? (v & kFlagVal) : 0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
    excl += part;
    if (incl) break;
    top -= 32;  // flags[0] always holds a prefix, so the walk ends
  }
  if (lane == 0) {
    if (!ok && status) atomicOr(status, ST_TIMEOUT);
    if (publish) atomicExch(&flags[item], kFlagIncl | (excl + agg));
  }
  return ok ? int64_t(excl) : -1;
}

}  // namespace gt
