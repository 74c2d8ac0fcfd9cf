"""Workloads that stand for what users of this library have it do.

Each case is a dict of plain values; its "kind" names the path:

  count    one document on the device -> its table (wc_count), answered with
           its top-k rows or exported whole
  host     one document in pinned host memory -> its table, exported whole
           (wc_count_host: the copy overlaps the count)
  round    a round of small documents counted per document (wc_count_batched),
           each answered with its top-k rows
  classes  documents in classes: per-class tables and each class's top words
           by class ratio (a plan, replayed)
  batch    many log-normal documents, counted per document through a plan,
           each answered with its top-k rows
  vocab    the sorted vocabulary of many log-normal documents (wc_batch_vocab:
           per-document tables, the reduce over them, word order and row ids)
  merge    tables of separate texts summed word by word (wc_merge)
  series   the two numeric sums of Sec. 4.2 of the paper (wc_series_sum)
  rows     row sums of a zero-padded count matrix (wc_row_sums)

Texts are Zipf draws from a seeded vocabulary, written on the GPU: the same
vocabulary sizes, exponents, word-length laws and separators as the recipes of
corpus/ (rank-correlated lengths, capitals, punctuation, newlines, digit runs).
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2206_05269_gb300 import wc

DEV = "cuda"

# vocabulary: size, Zipf exponent, word length = a + b ln(rank) + U(-jitter,
# jitter) (+ an exponential extra for some rare words), length limits; share of
# capitalised words, of separators with punctuation and of digit runs
VOCABS = {
    "tiny": dict(size=5_000, s=1.1, a=2.5, b=0.55, jitter=1.5, tail=0.0, tail_mean=0.0, lo=1, hi=12, cap=0.10,
                 punct=0.15, digits=0.0),
    "classes": dict(size=30_000, s=1.05, a=2.3, b=0.55, jitter=1.5, tail=0.0, tail_mean=0.0, lo=1, hi=14, cap=0.10,
                    punct=0.15, digits=0.0),
    "large": dict(size=1_000_000, s=1.0, a=0.2, b=0.6, jitter=2.0, tail=0.15, tail_mean=4.0, lo=1, hi=24, cap=0.20,
                  punct=0.12, digits=0.03),
    "batched": dict(size=200_000, s=1.1, a=1.5, b=0.55, jitter=1.5, tail=0.1, tail_mean=3.0, lo=1, hi=20, cap=0.10,
                    punct=0.15, digits=0.0),
    "served": dict(size=500_000, s=1.0, a=0.3, b=0.6, jitter=2.0, tail=0.15, tail_mean=4.0, lo=1, hi=22, cap=0.15,
                   punct=0.15, digits=0.0),
}
SEPARATORS = (b" ", b", ", b". ", b"; ", b" - ", b"\n", b" 17 ", b" 2024 ")


def listed():
    return [
        # the smallest served request: one short note, answered with its 100 most frequent words
        dict(name="served_2KB", kind="count", vocab="served", bytes=2_085, bits=32, topk=100, skew=3),
        # an ordinary served request: a book-sized document that arrives at an odd address
        dict(name="served_4MB", kind="count", vocab="served", bytes=3_999_971, bits=32, topk=100, skew=5),
        # the largest served request, its whole table kept
        dict(name="served_64MB", kind="count", vocab="served", bytes=64_000_000, bits=32, topk=0, skew=0),
        # the single-pass corpus count: 1 GB, a million-word vocabulary, 64-bit counts, the whole table out
        dict(name="corpus_1GB", kind="count", vocab="large", bytes=1_000_000_000, bits=64, topk=0, skew=0),
        # the same from host memory (end to end: text in, table out), a quarter of the size
        dict(name="host_256MB", kind="host", vocab="large", bytes=255_999_983, bits=64),
        # a round of short documents, as a serving loop admits them together: each answered with its top 100
        dict(name="round_200docs", kind="round", vocab="tiny", docs=200, words_lo=500, words_hi=3_000, topk=100),
        # the class study (Sec. 4.3): four classes of 250 speeches, class tables and the words each class uses most
        dict(name="classes_4x250", kind="classes", vocab="classes", classes=4, docs=1_000, words_lo=2_000,
             words_hi=8_000, topk=50),
        # the batched corpus: 100,000 documents through one plan, each answered with its top 100
        dict(name="batch_100k", kind="batch", vocab="batched", docs=100_000, topk=100),
        # 10,000 documents reduced to one sorted vocabulary with its counts
        dict(name="vocab_10k", kind="vocab", vocab="batched", docs=10_000),
        # the reduce across chunks: eight 16 MB chunks' tables summed
        dict(name="merge_8", kind="merge", vocab="large", tables=8, bytes=16_000_000),
        # the numeric MapReduce of Sec. 4.2 at its largest size, both series
        dict(name="series_1e8", kind="series", n=100_000_000),
        # the reduce of the hybrid pipeline of Sec. 3.3: 30,000 words by 1,000 documents
        dict(name="rows_30000x1000", kind="rows", rows=30_000, cols=1_000),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["count", "count", "count", "host", "round", "classes", "batch", "vocab", "merge", "series", "rows"])
    if kind == "count":
        return dict(kind=kind, vocab=rng.choice(["served", "large", "classes"]), bytes=_log_int(rng, 1_000, 600_000_000),
                    bits=rng.choice([32, 64]), topk=rng.choice([0, 0, 100]), skew=rng.randrange(16))
    if kind == "host":
        return dict(kind=kind, vocab=rng.choice(["served", "large"]), bytes=_log_int(rng, 1_000_000, 400_000_000),
                    bits=rng.choice([32, 64]))
    if kind == "round":
        lo = rng.randrange(50, 1_000)
        return dict(kind=kind, vocab=rng.choice(["tiny", "served"]), docs=_log_int(rng, 1, 1_000), words_lo=lo,
                    words_hi=lo + rng.randrange(1, 4_000), topk=rng.choice([10, 100]))
    if kind == "classes":
        lo = rng.randrange(200, 3_000)
        classes = rng.randrange(2, 9)
        return dict(kind=kind, vocab="classes", classes=classes, docs=classes * _log_int(rng, 10, 250), words_lo=lo,
                    words_hi=lo + rng.randrange(1, 6_000), topk=rng.choice([10, 50, 100]))
    if kind == "batch":
        return dict(kind=kind, vocab="batched", docs=_log_int(rng, 500, 100_000), topk=rng.choice([10, 100]))
    if kind == "vocab":
        return dict(kind=kind, vocab="batched", docs=_log_int(rng, 500, 30_000))
    if kind == "merge":
        return dict(kind=kind, vocab=rng.choice(["served", "large"]), tables=rng.randrange(2, 17),
                    bytes=_log_int(rng, 100_000, 30_000_000))
    if kind == "series":
        return dict(kind=kind, n=_log_int(rng, 1_000, 100_000_000))
    return dict(kind="rows", rows=_log_int(rng, 100, 30_000), cols=rng.randrange(1, 1_500))


# ---------------------------------------------------------------- inputs
def _generator(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _rand(g, n):
    return torch.rand(n, dtype=torch.float64, device=DEV, generator=g)


def _vocabulary(v, g):
    """(letters uint8 [size, hi], lengths int64 [size]) of a seeded vocabulary, most frequent word first."""
    n, hi = v["size"], v["hi"]
    t = v["a"] + v["b"] * torch.log(torch.arange(1, n + 1, dtype=torch.float64, device=DEV)) + \
        (_rand(g, n) * 2 - 1) * v["jitter"]
    if v["tail"]:
        extra = -torch.log1p(-_rand(g, n)) * v["tail_mean"]
        rare = (_rand(g, n) < v["tail"]) & (torch.arange(n, device=DEV) >= min(1000, n))
        t = torch.where(rare, t + extra, t)
    length = torch.floor(t + 0.5).clamp(v["lo"], hi).to(torch.int64)
    letters = torch.randint(0, 26, (n, hi), device=DEV, generator=g)
    for m in range(1, min(5, hi)):  # short words: all different, each length at most half used up
        at = torch.nonzero(length == m).flatten()
        room = 26 ** m // 2
        length[at[room:]] = m + 1
        at = at[:room]
        code = (torch.arange(at.numel(), device=DEV) * 7919 + int(17 * m)) % 26 ** m
        for j in range(m):
            letters[at, j] = code % 26
            code = code // 26
    return (letters + 97).to(torch.uint8), length


def _ids(v, g, n, weights=None):
    w = np.arange(1, v["size"] + 1, dtype=np.float64) ** -v["s"]
    if weights is not None:
        w = w * weights
    c = np.cumsum(w)
    cdf = torch.from_numpy(c / c[-1]).to(DEV)
    return torch.searchsorted(cdf, _rand(g, n), right=True).clamp_(max=v["size"] - 1)


def _write(v, g, letters, length, ids):
    """The text of the drawn words: (uint8 bytes, int64 [n + 1] first byte of each word)."""
    n = ids.numel()
    hi = letters.shape[1]
    sep_b = torch.zeros(len(SEPARATORS), 8, dtype=torch.uint8)
    for i, s in enumerate(SEPARATORS):
        sep_b[i, :len(s)] = torch.tensor(list(s), dtype=torch.uint8)
    sep_b = sep_b.to(DEV)
    sep_n = torch.tensor([len(s) for s in SEPARATORS], device=DEV)
    p = v["punct"]
    edges = np.cumsum([p * 0.5, p * 0.25, p * 0.15, p * 0.1, 1 / 14, v["digits"] / 2, v["digits"] / 2])
    sep = torch.bucketize(torch.rand(n, device=DEV, generator=g).double(), torch.from_numpy(edges).to(DEV))
    sep = torch.where(sep == len(SEPARATORS) - 1, 0, sep + 1)  # the rest: one space
    r = torch.rand(n, device=DEV, generator=g)
    cap = torch.where(r < v["cap"] / 2, 1, torch.where(r < v["cap"], hi, 0))  # letters in capitals: none, first, all
    off = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(length[ids] + sep_n[sep], 0, out=off[1:])
    total = int(off[-1])
    text = torch.empty(total, dtype=torch.uint8, device=DEV)
    flat, sflat = letters.reshape(-1), sep_b.reshape(-1)
    step = 16_000_000
    for t0 in range(0, n, step):
        t1 = min(n, t0 + step)
        b0, b1 = int(off[t0]), int(off[t1])
        lens = off[t0 + 1:t1 + 1] - off[t0:t1]
        tok = torch.repeat_interleave(torch.arange(t1 - t0, device=DEV), lens, output_size=b1 - b0)
        pos = torch.arange(b0, b1, device=DEV) - off[t0:t1][tok]
        i = ids[t0:t1][tok]
        ln = length[i]
        word = flat[i * hi + pos.clamp(max=hi - 1)]
        word = torch.where(pos < cap[t0:t1][tok], word - 32, word)
        other = sflat[sep[t0:t1][tok] * 8 + (pos - ln).clamp(0, 7)]
        text[b0:b1] = torch.where(pos < ln, word, other)
    return text, off


def _mean_bytes(v, length):
    w = np.arange(1, v["size"] + 1, dtype=np.float64) ** -v["s"]
    return float((w * length.cpu().numpy()).sum() / w.sum()) + 1.0 + v["punct"] + 2.0 * v["digits"]


def _text(v, g, nbytes, vocabulary=None):
    """nbytes of text."""
    letters, length = vocabulary or _vocabulary(v, g)
    n = int(nbytes / _mean_bytes(v, length) * 1.05) + 200
    text, _ = _write(v, g, letters, length, _ids(v, g, n))
    while text.numel() < nbytes:
        more, _ = _write(v, g, letters, length, _ids(v, g, n // 8 + 200))
        text = torch.cat([text, more])
    return text[:nbytes].clone()


def _skewed(text, skew):
    """The text at an address `skew` bytes past a 16-byte boundary."""
    buf = torch.empty(text.numel() + 32, dtype=torch.uint8, device=DEV)
    out = buf[skew:skew + text.numel()]
    out.copy_(text)
    return out


def _lognormal_docs(v, g, docs):
    """(text, offsets) of documents of log-normal byte length (median 2 KB, sigma 1.5, 1 KB to 1 MB), cut between words."""
    z = torch.randn(docs, dtype=torch.float64, device=DEV, generator=g)
    want = torch.exp(math.log(2048) + 1.5 * z).clamp(1024, 1 << 20).to(torch.int64)
    ends = torch.cumsum(want, 0)
    letters, length = _vocabulary(v, g)
    n = int(int(ends[-1]) / _mean_bytes(v, length) * 1.05) + 2_000
    text, off = _write(v, g, letters, length, _ids(v, g, n))
    first = torch.searchsorted(off, ends.clamp(max=text.numel()))
    cut = torch.cat([torch.zeros(1, dtype=torch.int64, device=DEV), off[first]])
    return text[:int(cut[-1])].clone(), cut


def _word_docs(v, g, docs, words_lo, words_hi, classes=0):
    """(text, offsets, classes) of documents of a uniform number of words; with classes, 200 words of each at 5 to 20
    times their rate."""
    count = torch.randint(words_lo, words_hi + 1, (docs,), device=DEV, generator=g)
    letters, length = _vocabulary(v, g)
    cls = torch.arange(docs, device=DEV) % max(classes, 1)
    n = int(count.sum())
    ids = _ids(v, g, n)
    if classes:
        owner = torch.repeat_interleave(cls, count, output_size=n)
        pick = torch.randperm(v["size"] - 100, device=DEV, generator=g)[:200 * classes].cpu().numpy() + 100
        rate = 5.0 + 15.0 * _rand(g, 200 * classes).cpu().numpy()
        for c in range(classes):
            w = np.ones(v["size"])
            w[pick[200 * c:200 * (c + 1)]] = rate[200 * c:200 * (c + 1)]
            mine = owner == c
            ids[mine] = _ids(v, g, int(mine.sum()), w)
    text, off = _write(v, g, letters, length, ids)
    first = torch.cat([torch.zeros(1, dtype=torch.int64, device=DEV), torch.cumsum(count, 0)])
    return text, off[first], cls.to(torch.int32)


class _Pinned:
    """Pinned host buffers for exported tables of at most `rows` rows and `nbytes` word bytes (what a table leaves
    unused stays zero)."""

    def __init__(self, rows, nbytes, bits):
        self.words = torch.zeros(nbytes + 16, dtype=torch.uint8).pin_memory()
        self.offsets = torch.zeros(rows + 1, dtype=torch.int64).pin_memory()
        self.counts = torch.zeros(rows, dtype=torch.int64 if bits == 64 else torch.int32).pin_memory()

    def take(self, table):
        n, nb = table.export_into(self.words, self.offsets, self.counts)
        return n, nb, self.words, self.offsets, self.counts


def _table_room(v, nbytes=None):
    """Rows and word bytes that no table over this vocabulary passes (a text may end in a cut word)."""
    rows = v["size"] + 16
    if nbytes is not None:
        rows = min(rows, nbytes // 2 + 1)
    return rows, min(rows * v["hi"], nbytes or rows * v["hi"])


def prepare(case, seed):
    g = _generator(seed)
    kind = case["kind"]
    st = dict(case=case)
    if kind == "series":
        st["counter"] = wc.Counter()
        st["n"] = case["n"] - 2 * (seed % 64)  # another seed is another length
        st["out"] = torch.zeros(2, dtype=torch.float64, device=DEV)
        return st
    if kind == "rows":
        rows, cols = case["rows"], case["cols"]
        m = torch.randint(1, 40, (rows, cols), dtype=torch.int32, device=DEV, generator=g)
        # row r holds one count per document with its word: nearly all for the frequent words, few for the rest
        filled = (cols / torch.arange(1, rows + 1, device=DEV).double().pow(0.5)).clamp(min=1.0)
        filled = (filled * (0.5 + _rand(g, rows))).clamp(max=cols).to(torch.int64)
        m *= (torch.arange(cols, device=DEV)[None, :] < filled[:, None]).to(torch.int32)
        st["matrix"], st["sums"] = m, torch.zeros(rows, dtype=torch.int64, device=DEV)
        return st
    v = VOCABS[case["vocab"]]
    if kind in ("count", "host"):
        text = _text(v, g, case["bytes"])
        st["counter"] = wc.Counter(count_bits=case["bits"])
        if kind == "count":
            st["text"] = _skewed(text, case["skew"])
        else:
            st["host"] = text.cpu().pin_memory()
            st["device"] = torch.empty(case["bytes"], dtype=torch.uint8, device=DEV)
        rows, room = _table_room(v, case["bytes"])
        if case.get("topk"):
            rows, room = case["topk"], case["topk"] * v["hi"]
        st["pinned"] = _Pinned(rows, room, case["bits"])
        return st
    if kind == "merge":
        vocabulary = _vocabulary(v, g)
        st["counter"] = wc.Counter()
        st["tables"] = [st["counter"].count_checked(_text(v, g, case["bytes"], vocabulary)) for _ in range(case["tables"])]
        st["pinned"] = _Pinned(*_table_room(v), 64)
        return st
    # documents
    if kind in ("round", "classes"):
        text, cut, cls = _word_docs(v, g, case["docs"], case["words_lo"], case["words_hi"], case.get("classes", 0))
    else:
        text, cut = _lognormal_docs(v, g, case["docs"])
    docs = case["docs"]
    st["text"], st["offsets"], st["h_offsets"] = text, cut, cut.cpu().numpy().astype(np.uint64)
    st["counter"] = wc.Counter(count_bits=32)
    if kind in ("round", "batch"):
        st["pinned"] = _Pinned(case["topk"] * docs, case["topk"] * docs * v["hi"], 32)
    elif kind == "classes":
        st["classes"] = cls
        st["pinned"] = [_Pinned(*_table_room(v), 32) for _ in range(case["classes"])]
    else:
        st["pinned"] = _Pinned(*_table_room(v), 64)
    if kind != "round":
        st["plan"] = st["counter"].plan(st["h_offsets"], case.get("classes", 0))
    return st


# ---------------------------------------------------------------- one pass
def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "series":
        s = torch.cuda.current_stream().cuda_stream
        for series in (wc.WC_SERIES_SQRT, wc.WC_SERIES_ALT_HARMONIC):
            wc.wc_series_sum(st["counter"].ctx, series, st["n"], st["out"].data_ptr() + 8 * series, s)
        return st["out"]
    if kind == "rows":
        wc.wc_row_sums(st["matrix"].data_ptr(), case["rows"], case["cols"], st["sums"].data_ptr(),
                       torch.cuda.current_stream().cuda_stream)
        return st["sums"]
    ctr = st["counter"]
    if kind in ("count", "host"):
        table = ctr.count_checked(st["text"]) if kind == "count" else ctr.count_host_checked(st["host"], out=st["device"])
        if case.get("topk"):
            top = ctr.topk(table, case["topk"])
            out = st["pinned"].take(top)
            top.free()
        else:
            out = st["pinned"].take(table)
        table.free()
        return out
    if kind == "merge":
        table = ctr.merge(st["tables"])
        out = st["pinned"].take(table)
        table.free()
        return out
    if kind == "round":
        batch = ctr.count_batched_checked(st["text"], st["offsets"], st["h_offsets"])
    else:
        batch = st["plan"].run(st["text"], st["offsets"], st.get("classes"))
        if batch.status() != wc.WC_OK:
            raise RuntimeError("batched count: " + wc.wc_last_error(ctr.ctx))
    if kind == "classes":
        out = []
        for c in range(case["classes"]):
            idx, cin, cout = wc.wc_class_ratio_topk(ctr.ctx, batch.handle, c, case["topk"],
                                                    torch.cuda.current_stream().cuda_stream)
            out.append((np.stack([idx, cin, cout]),) + st["pinned"][c].take(batch.table(wc.WC_TABLE_CLASS, c)))
        return out
    if kind == "vocab":
        return st["pinned"].take(batch.vocab())
    top, first, sizes = batch.topk(case["topk"])
    out = (first, sizes) + st["pinned"].take(top)
    if kind == "round":
        batch.free()
    return out


# ---------------------------------------------------------------- floors and exact values
def _distinct(v, tokens):
    """Expected distinct words of so many Zipf draws."""
    w = np.arange(1, v["size"] + 1, dtype=np.float64) ** -v["s"]
    return float(-np.expm1(tokens * np.log1p(-w / w.sum())).sum())


def _row_bytes(v, rows, bits):
    return rows * (v["a"] + v["b"] * math.log(v["size"]) + 8 + bits / 8)


def work(case):
    """Bytes: the text (tables, matrix) read once, the result written once; no floating-point work but the series' terms."""
    kind = case["kind"]
    if kind == "series":  # a square root, or a division and a sign, and an addition a term
        return {"bytes": 16, "flops": 4.0 * case["n"]}
    if kind == "rows":
        return {"bytes": 4.0 * case["rows"] * case["cols"] + 8.0 * case["rows"], "flops": 0}
    v = VOCABS[case["vocab"]]
    word = v["a"] + v["b"] * 5 + 1.3
    if kind in ("count", "host"):
        rows = _distinct(v, case["bytes"] / word)
        if case.get("topk"):
            rows = min(rows, case["topk"])
        return {"bytes": case["bytes"] + _row_bytes(v, rows, case["bits"]), "flops": 0}
    if kind == "merge":
        one = _distinct(v, case["bytes"] / word)
        return {"bytes": 28.0 * one * case["tables"] + _row_bytes(v, _distinct(v, case["tables"] * case["bytes"] / word), 64),
                "flops": 0}
    docs = case["docs"]
    if kind in ("round", "classes"):
        words = (case["words_lo"] + case["words_hi"]) / 2
        if kind == "round":
            rows = docs * _row_bytes(v, min(case["topk"], _distinct(v, words)), 32) + 12 * docs
        else:
            rows = case["classes"] * (_row_bytes(v, _distinct(v, words * docs / case["classes"]), 32) + 24 * case["topk"])
        return {"bytes": docs * words * word + rows, "flops": 0}
    if kind == "batch":
        return {"bytes": docs * 6_480 + docs * (12 + _row_bytes(v, min(case["topk"], _distinct(v, 400)), 32)), "flops": 0}
    return {"bytes": docs * 6_480 + _row_bytes(v, _distinct(v, docs * 1_200), 64), "flops": 0}


def exact(case, seed):
    """The series' sums of correctly rounded terms, exactly, and the row sums; counts are whole numbers."""
    if case["kind"] == "rows":
        return prepare(case, seed)["matrix"].to(torch.int64).sum(1)
    if case["kind"] != "series":
        return None
    n = case["n"] - 2 * (seed % 64)
    sums = []
    for series, (b0, b1) in enumerate(((26, 52), (40, 80))):  # a term = hi / 2^b0 + lo / 2^b1, hi and lo whole
        hi = lo = 0
        for i0 in range(1, n + 1, 1 << 20):
            i = np.arange(i0, min(n + 1, i0 + (1 << 20)), dtype=np.float64)
            t = np.sqrt(i) if series == 0 else 1.0 / i
            h = np.floor(t * 2.0 ** b0)
            d = (t - h * 2.0 ** -b0) * 2.0 ** b1
            if series:
                sign = np.where(i % 2 == 1, 1, -1)
                hi += int((h.astype(np.int64) * sign).sum())
                lo += int((d.astype(np.int64) * sign).sum())
            else:
                hi += int(h.astype(np.int64).sum())
                lo += int(d.astype(np.int64).sum())
        whole = (hi << (b1 - b0)) + lo
        sums.append(whole / (1 << b1))
    return np.array(sums, dtype=np.float64)
