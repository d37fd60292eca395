"""Performance cases of the engine: what a program that analyses compressed
corpora asks of it, from one small file to the 100M-token nested corpus.

The corpora are the shapes of ``paper_2106_06889_gb300.corpus.CONFIGS`` and of
the serving set (Zipf words, repeated passages, nested phrases, many files),
drawn here on the GPU from a seed and compressed by the package's Sequitur.
Corpora above 4M tokens are compressed as 16 pieces whose grammars are
concatenated (``sequitur_sharded``, as ``load_config`` does for its largest
corpus), which keeps the preparation to seconds.
"""
import ctypes
import functools
import math
from concurrent.futures import ThreadPoolExecutor

import numpy as np
import torch

from paper_2106_06889_gb300 import binding as B
from paper_2106_06889_gb300.corpus import sequitur, sequitur_sharded


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------

def _case(op, kind, tokens, vocab, zipf, files=1, lo=0, hi=0, param=0):
    """``lo`` / ``hi``: range of file lengths (their proportions where ``kind`` is
    "files", whose total is ``tokens``); ``param``: the option of the analytic."""
    return {"op": op, "kind": kind, "tokens": tokens, "vocab": vocab, "zipf": zipf, "files": files, "lo": lo,
            "hi": hi, "param": param}


def listed():
    return [
        # one small document, its words counted: the shortest query there is
        dict(_case("count", "passages", 200_000, 20_000, 1.1), name="count_small"),
        # one large file with nested repeats (deep rule DAG), its words counted
        dict(_case("count", "nested", 100_000_000, 1_000_000, 1.05), name="count_large"),
        # the headline step of bench.py: word count, inverted index and term
        # vector of 64 files sharing one grammar, as a plan replayed per step
        dict(_case("files_plan", "files", 50_000_000, 500_000, 1.0, 64, 10_000, 2_000_000), name="files64_plan"),
        # TF-IDF and the 20 most frequent words of an odd number of mid-sized files
        dict(_case("vectors", "files", 6_000_000, 300_007, 1.05, 37, 10_000, 2_000_000, 20), name="vectors_mid"),
        # 3-word count of the small document: a chain of short kernels
        dict(_case("sequence", "passages", 200_000, 20_000, 1.1), name="seq_small"),
        # the nested corpus' step of bench.py: 3-word count and words sorted by count
        dict(_case("sequence_sort", "nested", 100_000_000, 1_000_000, 1.05, param=1), name="seq_sort_large"),
        # 3-word counts of every file of a 64-file corpus (top-down strategy)
        dict(_case("sequence_files", "files", 8_000_000, 500_000, 1.0, 64, 10_000, 2_000_000), name="seq_files"),
        # term vector and inverted index of many files of 1k-50k words (bottom-up strategy)
        dict(_case("index", "many", 25_000_000, 200_000, 1.1, 2_000, 1_000, 50_000), name="index_many"),
        # 3-word ranked inverted index of many short files (each fits one CTA)
        dict(_case("ranked", "many", 10_000_000, 200_000, 1.1, 8_000, 100, 5_000, 3), name="ranked_short"),
        # word co-occurrence of a serving-sized corpus
        dict(_case("cooccurrence", "files", 4_000_000, 1_000_000, 1.1, 9, 10_000, 2_000_000), name="cooc_mid"),
        # a new corpus from host memory: load, word count and inverted index, free
        dict(_case("ingest", "files", 8_000_000, 1_000_000, 1.1, 13, 10_000, 2_000_000), name="ingest_mid"),
        # the serving mix of bench.py (40% word count, 30% inverted index, 30%
        # 3-word count) over four resident corpora, 16 requests at once
        dict(_case("serve", "files", 6_000_000, 1_000_000, 1.1, 12, 10_000, 2_000_000, 16), name="serve_mix"),
    ]


# per op: corpus kinds, tokens, vocabulary and number of files its draws range over
_RANGES = {
    "count": (("passages", "nested", "files"), (50_000, 64_000_000), (5_000, 1_000_000), (2, 64)),
    "files_plan": (("files",), (300_000, 32_000_000), (20_000, 500_000), (2, 64)),
    "vectors": (("files",), (200_000, 8_000_000), (20_000, 1_000_000), (2, 64)),
    "sequence": (("passages", "nested"), (50_000, 16_000_000), (5_000, 1_000_000), (1, 1)),
    "sequence_sort": (("nested", "files"), (1_000_000, 64_000_000), (20_000, 1_000_000), (2, 64)),
    "sequence_files": (("files",), (200_000, 8_000_000), (20_000, 500_000), (2, 64)),
    "index": (("many",), (500_000, 25_000_000), (20_000, 400_000), (65, 4_000)),
    "ranked": (("many",), (300_000, 10_000_000), (20_000, 400_000), (65, 8_000)),
    "cooccurrence": (("files", "nested"), (200_000, 6_000_000), (20_000, 1_000_000), (2, 64)),
    "ingest": (("files", "nested"), (300_000, 8_000_000), (20_000, 1_000_000), (2, 64)),
    "serve": (("files",), (1_000_000, 6_000_000), (200_000, 1_000_000), (2, 64)),
}


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    op = rng.choice(sorted(_RANGES))
    kinds, tokens, vocab, files = _RANGES[op]
    kind = rng.choice(kinds)
    n = log(*tokens)
    c = _case(op, kind, n, log(*vocab), round(rng.uniform(1.0, 1.2), 3))
    if kind == "files":
        c.update(files=log(*files), lo=10_000, hi=2_000_000)
    elif kind == "many":
        # lengths log-uniform over a factor of 50, as in the many-files
        # configurations: short files and long ones, by their mean
        c["files"] = max(files[0], min(log(*files), n // 100))
        mean = n / c["files"]
        c.update(lo=max(1, int(mean / 12.5)), hi=max(2, int(mean * 4)))
    c["param"] = {"vectors": rng.choice([5, 20, 100]), "sequence_sort": rng.choice([0, 1]),
                  "ranked": rng.choice([1, 3, 3]), "serve": rng.choice([8, 12, 16])}.get(op, 0)
    return c


# ---------------------------------------------------------------------------
# corpora
# ---------------------------------------------------------------------------

def _zipf_draw(gen, n, cdf, perm):
    out = torch.empty(n, dtype=torch.int32, device="cuda")
    for a in range(0, n, 1 << 25):  # pieces: the float64 draws of 100M words need not exist at once
        b = min(n, a + (1 << 25))
        u = torch.rand(b - a, generator=gen, device="cuda", dtype=torch.float64)
        out[a:b] = perm[torch.searchsorted(cdf, u, right=True).clamp_(max=cdf.shape[0] - 1)]
    return out.cpu().numpy()


def _pieces(rng, gen, case, cdf, perm):
    """The repeated passages to insert, in insertion order."""
    n = case["tokens"]
    if case["kind"] == "passages":  # 20% of the text: passages of 200 words, each four times
        pool = _zipf_draw(gen, max(1, n // 4000) * 200, cdf, perm).reshape(-1, 200)
        return [p for p in pool for _ in range(4)]
    if case["kind"] == "files":  # 5% of the text from a shared pool of 500 passages
        pool = _zipf_draw(gen, 500 * 200, cdf, perm).reshape(-1, 200)
        return [pool[i] for i in rng.integers(0, 500, size=n // 4000)]
    if case["kind"] == "nested":  # half of the text: phrases of phrases, six levels of four
        levels = [list(_zipf_draw(gen, 4096 * 16, cdf, perm).reshape(-1, 16))]
        for _ in range(6):
            prev = levels[-1]
            levels.append([np.concatenate([prev[i] for i in rng.integers(0, len(prev), size=4)]) for _ in range(256)])
        pieces, got = [], 0
        while got < n // 2:
            lv = levels[int(rng.integers(1, 7))]
            p = lv[int(rng.integers(0, len(lv)))]
            if got + p.shape[0] > n // 2:
                break
            pieces.append(p)
            got += p.shape[0]
        return pieces
    return []


def _text(case, seed):
    """(tokens int32, file lengths int64): seeded, the same wherever it is drawn."""
    rng = np.random.default_rng([int(seed), 6889])
    gen = torch.Generator(device="cuda").manual_seed(int(rng.integers(1 << 62)))
    V, F, n = case["vocab"], case["files"], case["tokens"]
    w = np.arange(1, V + 1, dtype=np.float64) ** -case["zipf"]
    cdf = torch.from_numpy(np.cumsum(w) / w.sum()).cuda()
    perm = torch.from_numpy(rng.permutation(V).astype(np.int32)).cuda()
    pieces = _pieces(rng, gen, case, cdf, perm)
    lens = np.full(1, 1.0) if F == 1 else np.exp(rng.uniform(np.log(case["lo"]), np.log(case["hi"]), size=F))
    base_n = n - sum(p.shape[0] for p in pieces)
    lens = np.maximum(np.round(lens / lens.sum() * base_n), 1).astype(np.int64)
    base = _zipf_draw(gen, int(lens.sum()), cdf, perm)
    if not pieces:
        return base, lens
    at = np.sort(rng.integers(0, base.shape[0] + 1, size=len(pieces)))
    pieces = [pieces[k] for k in rng.permutation(len(pieces))]
    parts, last = [], 0
    for p, piece in zip(at, pieces):
        parts += [base[last:p], piece]
        last = p
    parts.append(base[last:])
    # a piece inserted at position p belongs to the file holding word p (the last one at the end)
    file_of = np.minimum(np.searchsorted(np.cumsum(lens), at, side="right"), F - 1)
    lens = lens + np.bincount(file_of, [p.shape[0] for p in pieces], F).astype(np.int64)
    return np.concatenate(parts).astype(np.int32), lens


def _compress(tokens, lens, V):
    if tokens.shape[0] <= 4_000_000:
        return sequitur(tokens, lens, V)
    return sequitur_sharded(tokens, lens, V, 16)


def _serve_texts(case, seed):
    """Four corpora of tokens/4 to tokens words."""
    return [_text(dict(case, tokens=max(1000, int(case["tokens"] * 4.0 ** (-i / 3.0))), files=max(2, case["files"] - i)),
                  int(seed) * 4 + i) for i in range(4)]


# ---------------------------------------------------------------------------
# preparation
# ---------------------------------------------------------------------------

@functools.lru_cache(maxsize=None)
def _ctx():
    return B.gt_create(0)


_II, _TV, _SEQ = ("offsets", "file"), ("offsets", "word", "count"), ("key", "count")
_RANKED = ("offsets", "key", "file", "count")
_TYPES = {"word": ("<i4", torch.int32), "file": ("<i4", torch.int32), "tfidf": ("<f8", torch.float64)}
_WHOLE = ("<i8", torch.int64)  # offsets, keys and counts

# the result fields that an op's pass returns, per result
_FIELDS = {"count": [], "files_plan": [_II, _TV], "vectors": [_TV + ("tfidf",), _TV], "sequence": [_SEQ],
           "sequence_sort": [_SEQ, ("word", "count")], "sequence_files": [("file",) + _SEQ], "index": [_TV, _II],
           "ranked": [_RANKED], "cooccurrence": [_SEQ], "ingest": [_II]}


def _requests(n):
    """(corpus, kind) of n requests: 40% word count, 30% inverted index, 30% 3-word count."""
    return [(i % 4, "wiswiwswsi"[i % 10]) for i in range(n)]


def _fields(case):
    if case["op"] == "serve":
        return [() if k == "w" else _II if k == "i" else _SEQ for _, k in _requests(case["param"])]
    return _FIELDS[case["op"]]


def _room(case, field):
    """Values a field can hold whatever the seed: no analytic has more rows than the text has words."""
    return case["tokens"] + 2 * case["files"] + (max(case["vocab"], case["files"]) + 1 if field == "offsets" else 0)


class _View:
    """A library-owned device buffer, for torch.as_tensor."""

    def __init__(self, ptr, n, typestr):
        self.__cuda_array_interface__ = {"shape": (n,), "typestr": typestr, "data": (ptr, False), "version": 3,
                                         "strides": None}


class _State:
    """Grammars, handles and buffers a user's program keeps between queries."""

    def __init__(self, case):
        self.case, self.grammars, self.plan, self.server = case, [], None, None
        # results are copied into buffers of the program's own, as large as a
        # field can get for this case; what a result does not fill stays zero
        self.buffers = [{f: torch.zeros(_room(case, f), dtype=_TYPES.get(f, _WHOLE)[1], device="cuda") for f in fields}
                        for fields in _fields(case)]

    def keep(self, i, field, ptr, n):
        buf = self.buffers[i][field]
        if n:
            buf[:n].copy_(torch.as_tensor(_View(ptr, n, _TYPES.get(field, _WHOLE)[0]), device="cuda"))
        return buf

    def take(self, *results):
        """The fields of every result, which are then freed (None: nothing to take)."""
        out = []
        for i, r in enumerate(results):
            if r is not None:
                out += [self.keep(i, f, *B.gt_result_view(r, f)) for f in self.buffers[i]]
                B.gt_free_result(r)
        return out

    def __del__(self):
        if self.server is not None:
            B.gt_server_destroy(self.server)
        if self.plan is not None:
            B.gt_plan_destroy(self.plan)
        for g in self.grammars:
            B.gt_free_grammar(g)


def prepare(case, seed):
    st = _State(case)
    V, op = case["vocab"], case["op"]
    if op == "serve":
        texts = _serve_texts(case, seed)
        with ThreadPoolExecutor(4) as ex:
            gs = list(ex.map(lambda t: sequitur(t[0], t[1], V), texts))
    else:
        gs = [_compress(*_text(case, seed), V)]
    if op == "ingest":  # host arrays in pinned memory, as a loading program holds them
        st.host = gs[0]
        for k in ("rule_off", "sym", "file_off"):
            setattr(st.host, k, torch.from_numpy(getattr(st.host, k)).pin_memory().numpy())
        return st
    st.grammars = [B.gt_load_grammar(_ctx(), g) for g in gs]
    g = st.grammars[0]
    if op in ("count", "files_plan"):
        st.counts = torch.empty(V, dtype=torch.int64, device="cuda")
    if op == "files_plan":
        st.plan = B.gt_plan_create(_ctx(), [(g, B.GT_Q_INVERTED_INDEX, 0, None), (g, B.GT_Q_TERM_VECTOR, 0, None),
                                            (g, B.GT_Q_WORD_COUNT, 0, st.counts)])
    if op == "serve":
        kinds = {"w": B.GT_Q_WORD_COUNT, "i": B.GT_Q_INVERTED_INDEX, "s": B.GT_Q_SEQUENCE_COUNT}
        st.requests = [(st.grammars[c], kinds[k], 0,
                        torch.empty(V, dtype=torch.int64, device="cuda") if k == "w" else None)
                       for c, k in _requests(case["param"])]
        st.server = B.gt_server_create(_ctx(), 8, 0)
    return st


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------

def _plan_field(st, i, field):
    p, n = ctypes.c_void_p(), ctypes.c_int64()
    rc = B.lib().gt_plan_result(st.plan.handle, i, field.encode(), ctypes.byref(p), ctypes.byref(n))
    if rc != B.GT_OK:
        raise B.GtError(rc, B.lib().gt_last_error(_ctx().handle).decode())
    return st.keep(i, field, p.value, n.value)


def run(st):
    op, param = st.case["op"], st.case["param"]
    g = st.grammars[0] if st.grammars else None
    if op == "count":
        B.gt_word_count(g, st.counts)
        return [st.counts]
    if op == "files_plan":
        B.gt_plan_launch(st.plan)
        return [st.counts] + [_plan_field(st, i, f) for i in (0, 1) for f in st.buffers[i]]
    if op == "vectors":
        return st.take(*B.gt_run_batch(_ctx(), [(g, B.GT_Q_TFIDF, 0, None), (g, B.GT_Q_TERM_VECTOR, param, None)]))
    if op == "sequence":
        return st.take(B.gt_sequence_count(g, 0))
    if op == "sequence_sort":
        return st.take(*B.gt_run_batch(_ctx(), [(g, B.GT_Q_SEQUENCE_COUNT, 0, None), (g, B.GT_Q_SORT, param, None)]))
    if op == "sequence_files":
        return st.take(B.gt_sequence_count(g, 1))
    if op == "index":
        return st.take(*B.gt_run_batch(_ctx(), [(g, B.GT_Q_TERM_VECTOR, 0, None), (g, B.GT_Q_INVERTED_INDEX, 0, None)]))
    if op == "ranked":
        return st.take(B.gt_ranked_index(g, param))
    if op == "cooccurrence":
        return st.take(B.gt_cooccurrence(g))
    if op == "ingest":
        counts = torch.empty(st.case["vocab"], dtype=torch.int64, device="cuda")
        h = B.gt_load_grammar(_ctx(), st.host)
        out = B.gt_run_batch(_ctx(), [(h, B.GT_Q_INVERTED_INDEX, 0, None), (h, B.GT_Q_WORD_COUNT, 0, counts)])
        out = [counts] + st.take(*out)
        B.gt_free_grammar(h)
        return out
    tickets = [B.gt_submit(st.server, [q]) for q in st.requests]
    results = [B.gt_poll(st.server, t, 1)[0][0] for t in tickets]
    return [q[3] for q in st.requests if q[3] is not None] + st.take(*results)


# ---------------------------------------------------------------------------
# the work of a pass, and its exact outputs
# ---------------------------------------------------------------------------

def _distinct(n, V, s):
    """Expected number of distinct words among n Zipf draws."""
    p = np.arange(1, V + 1, dtype=np.float64) ** -s
    return float((1 - np.exp(-n * p / p.sum())).sum())


def work(case):
    """Bytes: the grammar's arrays read once and the outputs written once.  How far a
    text compresses and how many of its windows differ depend on the draw; the
    shares used here are those of the listed corpora (within about a tenth)."""
    op, n, V, s, F = (case[k] for k in ("op", "tokens", "vocab", "zipf", "files"))
    fresh = n * {"passages": 0.85, "files": 0.95, "nested": 0.52}.get(case["kind"], 1.0)  # words outside repeats
    grammar = 4 * 0.8 * fresh + 8 * 0.035 * fresh + 8 * F  # 0.8 symbols and 0.035 rules per fresh word
    windows, pairs = 0.75 * fresh, F * _distinct(n / F, V, s)  # distinct 3-word keys; (file, word) pairs
    ii, tv, seq = 8 * V + 4 * pairs, 8 * F + 12 * pairs, 16 * windows
    out = {"count": 8 * V, "files_plan": 8 * V + ii + tv, "vectors": tv + 8 * pairs + 12 * F * case["param"],
           "sequence": seq, "sequence_sort": seq + 12 * _distinct(n, V, s), "sequence_files": 20 * 0.9 * fresh,
           "index": tv + ii, "cooccurrence": 16 * 0.9 * fresh, "ingest": 8 * V + ii,
           "ranked": 28 * 0.9 * fresh if case["param"] == 3 else 28 * pairs}
    # operations: one count, weight or comparison per symbol read and row written
    if op == "serve":  # the requests' mean corpus is 0.56 of the largest
        b = case["param"] * (0.56 * grammar + 0.4 * 8 * V + 0.3 * 0.56 * ii + 0.3 * 0.56 * seq)
        return {"bytes": int(b), "flops": int(case["param"] * 0.56 * n)}
    return {"bytes": int(grammar + out[op]), "flops": int(2 * fresh)}


class _Exact:
    """The analytics of one text by their definitions, in 64-bit torch."""

    def __init__(self, text, V):
        self.tok = torch.from_numpy(text[0]).cuda().long()
        lens = torch.from_numpy(np.asarray(text[1])).cuda()
        self.V, self.F = V, lens.shape[0]
        self.file = torch.repeat_interleave(torch.arange(self.F, device="cuda"), lens)

    def counts(self):
        return torch.bincount(self.tok, minlength=self.V)

    def sort(self, order):
        c = self.counts()
        w = torch.nonzero(c).flatten()
        if order:
            w = w[torch.sort(c[w], descending=True, stable=True).indices]
        return [w.int(), c[w]]

    @staticmethod
    def offsets(group, n):
        z = torch.zeros(1, dtype=torch.int64, device="cuda")
        return torch.cat([z, torch.cumsum(torch.bincount(group, minlength=n), 0)])

    def pairs(self):
        """(file, word, count) in (file, word) order."""
        k, c = torch.unique(self.file * self.V + self.tok, return_counts=True)
        return k // self.V, k % self.V, c

    def term_vector(self, top=0):
        f, w, c = self.pairs()
        if top:
            o = torch.sort(c, descending=True, stable=True).indices
            o = o[torch.sort(f[o], stable=True).indices]
            f, w, c = f[o], w[o], c[o]
            keep = torch.arange(f.shape[0], device="cuda") - self.offsets(f, self.F)[f] < top
            f, w, c = f[keep], w[keep], c[keep]
        return [self.offsets(f, self.F), w.int(), c]

    def tfidf(self):
        f, w, c = self.pairs()
        idf = torch.log(self.F / torch.bincount(w, minlength=self.V).double())
        return [self.offsets(f, self.F), w.int(), c, c.double() * idf[w]]

    def inverted_index(self):
        f, w, _ = self.pairs()
        o = torch.sort(w, stable=True).indices
        return [self.offsets(w, self.V), f[o].int()]

    def windows(self):
        t, inside = self.tok, self.file[2:] == self.file[:-2]
        return (t[:-2] << 42 | t[1:-1] << 21 | t[2:])[inside], self.file[2:][inside]

    def sequence(self):
        return list(torch.unique(self.windows()[0], return_counts=True))

    def file_rows(self, n):
        """(file, key, count) in (file, key) order; n = 3: windows, 1: words."""
        if n == 1:
            return self.pairs()
        k, f = self.windows()
        u, inv = torch.unique(k, return_inverse=True)
        fu, c = torch.unique(f << 32 | inv, return_counts=True)
        return fu >> 32, u[fu & 0xffffffff], c

    def sequence_files(self):
        f, k, c = self.file_rows(3)
        return [f.int(), k, c]

    def ranked(self, n):
        f, k, c = self.file_rows(n)
        o = torch.sort(c, descending=True, stable=True).indices
        o = o[torch.sort(k[o], stable=True).indices]
        u, per = torch.unique(k, return_counts=True)
        return [torch.cat([torch.zeros_like(per[:1]), torch.cumsum(per, 0)]), u, f[o].int(), c[o]]

    def cooccurrence(self):
        t, f = self.tok, self.file
        one = (t[:-1] << 21 | t[1:])[f[:-1] == f[1:]]
        two = (t[:-2] << 21 | t[2:])[f[:-2] == f[2:]]
        return list(torch.unique(torch.cat([one, two]), return_counts=True))


def exact(case, seed):
    op, V, param = case["op"], case["vocab"], case["param"]
    if op == "serve":
        xs = [_Exact(t, V) for t in _serve_texts(case, seed)]
        req = [(xs[c], k) for c, k in _requests(param)]
        counts = [x.counts() for x, k in req if k == "w"]
        results = [[] if k == "w" else x.inverted_index() if k == "i" else x.sequence() for x, k in req]
    else:
        x = _Exact(_text(case, seed), V)
        counts = [x.counts()] if op in ("count", "files_plan", "ingest") else []
        results = {"count": lambda: [],
                   "files_plan": lambda: [x.inverted_index(), x.term_vector()],
                   "vectors": lambda: [x.tfidf(), x.term_vector(param)],
                   "sequence": lambda: [x.sequence()],
                   "sequence_sort": lambda: [x.sequence(), x.sort(param)],
                   "sequence_files": lambda: [x.sequence_files()],
                   "index": lambda: [x.term_vector(), x.inverted_index()],
                   "ranked": lambda: [x.ranked(param)],
                   "cooccurrence": lambda: [x.cooccurrence()],
                   "ingest": lambda: [x.inverted_index()]}[op]()
    return counts + [torch.nn.functional.pad(v, (0, _room(case, f) - v.shape[0]))
                     for fields, values in zip(_fields(case), results) for f, v in zip(fields, values)]
