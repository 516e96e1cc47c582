"""Performance cases of the batched RAMBO query and insertion: the work a program
using this package has it do, through its public calls.

Inputs are synthetic genomes drawn on the GPU from the case's seed: documents are
mutated copies of uniform seed genomes (families of about 50), queries are
substrings of documents with 0.1% read errors or uniform sequences, as in the
workloads of paper_1910_04358_gb300/synth.py.  Every output is an answer bit
mask, whole numbers that are either right or wrong, so there is no exact().
"""
import math

import numpy as np
import torch

from paper_1910_04358_gb300 import autotune, rambo

# Tunings that ship with the package (autotune's cache), by their keys there.
TUNED = {
    "medium": "K1000_B32_R4_m67108864_eta2_k31_n1010000_kpq10",
    "large": "K10000_B100_R5_m536870912_eta2_k31_n100000_kpq2480",
    "stream": "K100000_B316_R6_m268435456_eta2_k31_n10000_stream",
}

# Geometry (K documents, B buckets, R repetitions, m positions) of the package's workloads.
MEDIUM = dict(K=1000, B=32, R=4, m=1 << 26, eta=2, k=31, docs=1000, doc_len=1_000_000)
LARGE = dict(K=10_000, B=100, R=5, m=1 << 29, eta=2, k=31, docs=10_000, doc_len=500_000)
# the large geometry at 1/8 of the positions and document length (same filling, 4 GiB)
EIGHTH = dict(LARGE, m=1 << 26, doc_len=62_500)
# the streaming geometry at a quarter of the positions and documents held (16 GiB)
STREAM = dict(K=100_000, B=316, R=6, m=1 << 26, eta=2, k=31, docs=25_000, doc_len=50_000)


def listed():
    return [
        # one interactive lookup: a handful of k-mers, nothing to hide a launch behind
        dict(name="kmers_few", op="kmers", K=1000, B=32, R=4, m=1 << 22, eta=2, k=31, docs=1000,
             doc_len=60_000, tuning="", n_kmers=32, n_seqs=0),
        # short reads against a small index that stays in L2 (the tiny workload)
        dict(name="seqs_tiny", op="seqs", K=100, B=10, R=2, m=1 << 20, eta=2, k=31, docs=100,
             doc_len=20_000, tuning="", n_kmers=0, n_seqs=1000, lo=100, hi=100, shape="uniform"),
        # one batch of a server: 256 requests, log-normal lengths, at byte boundaries
        dict(name="serve_256", op="ranges", **EIGHTH, tuning="large", n_kmers=0, n_seqs=256, lo=31,
             hi=10_000, shape="lognormal"),
        # single-term queries, the paper's own measure, over 1,000 documents, default knobs
        dict(name="kmers_medium", op="kmers", **MEDIUM, tuning="", n_kmers=1_000_000, n_seqs=0),
        # single-term queries over 10,000 documents: 1,252-byte answers
        dict(name="kmers_10k_docs", op="kmers", **EIGHTH, tuning="", n_kmers=100_000, n_seqs=0),
        # the paper's 500-file parameters with its kind of m (no power of two), short ragged reads
        dict(name="reads_odd_m", op="seqs", K=500, B=60, R=3, m=200_000_000, eta=2, k=31, docs=500,
             doc_len=2_000_000, tuning="", n_kmers=0, n_seqs=20_011, lo=31, hi=301, shape="uniform"),
        # both kinds in one call, device buffers (the medium workload)
        dict(name="batch_medium", op="batch", **MEDIUM, tuning="medium", n_kmers=1_000_000,
             n_seqs=10_000, lo=1000, hi=1000, shape="uniform"),
        # the same call with the caller's page-locked host buffers
        dict(name="host_medium", op="host", **MEDIUM, tuning="medium", n_kmers=1_000_000,
             n_seqs=10_000, lo=1000, hi=1000, shape="uniform"),
        # the large workload: 10^5 sequences against a 32 GiB index
        dict(name="seqs_large", op="seqs", **LARGE, tuning="large", n_kmers=0, n_seqs=100_000, lo=31,
             hi=5000, shape="uniform"),
        # a streaming epoch: 1,000 documents arrive, then 10,000 queries
        dict(name="stream_epoch", op="epoch", **STREAM, tuning="stream", n_kmers=0, n_seqs=10_000,
             lo=31, hi=2000, shape="uniform", epoch_docs=1000),
        # building the medium index (10^9 k-mers), then looking at it
        dict(name="build_medium", op="build", **MEDIUM, tuning="medium", n_kmers=100_000, n_seqs=0),
        # documents of words at the paper's Wiki-dump parameters: 1,000 short queries
        dict(name="words_wiki", op="words", K=17_618, B=1000, R=2, m=200_000, eta=2, k=31, docs=17_618,
             doc_len=50, tuning="", n_kmers=0, n_seqs=1000, lo=1, hi=4, shape="uniform"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _group_bytes(case):
    """Bytes of one position group as the index lays it out."""
    raw = (case["R"] * case["B"] + 31) // 32 * 4
    if raw > 512:
        return (raw + 511) // 512 * 512
    return 1 << (raw - 1).bit_length()


def draw(rng):
    op = rng.choice(["kmers", "kmers", "seqs", "seqs", "seqs", "ranges", "batch", "host", "epoch", "build",
                     "words"])
    c = dict(op=op, k=rng.choice([21, 25, 31, 31, 31]), eta=rng.choice([1, 2, 2, 2, 3, 4]), tuning="")
    c["K"] = _log(rng, 40, 30_000)
    c["B"] = rng.choice([7, 10, 15, 27, 32, 50, 60, 64, 100, 128, 200, 316])
    c["R"] = rng.choice([2, 3, 3, 4, 5, 6])
    words = (c["K"] + 31) // 32
    if op == "words":
        c.update(B=_log(rng, 100, 5000), R=rng.choice([2, 3]), m=_log(rng, 20_000, 400_000), docs=c["K"],
                 doc_len=rng.randint(20, 60), n_kmers=0, n_seqs=_log(rng, 10, 5000), lo=1,
                 hi=rng.randint(1, 8), shape="uniform")
        return c
    m = _log(rng, 1 << 14, min(1 << 26, (6 << 30) // _group_bytes(c)))
    c["m"] = 1 << (m.bit_length() - 1) if rng.random() < 0.5 else m
    c["docs"] = c["K"]
    # documents that fill about a third of the bits of their buckets
    fill = int(0.35 * c["m"] * c["B"] / (c["K"] * c["eta"]))
    c["doc_len"] = max(200, min(fill, 500_000, 1_000_000_000 // c["K"]))
    most = min(1_000_000, (192 << 20) // (4 * words))  # answers of at most 192 MiB
    c["n_kmers"] = _log(rng, 1, most) if op in ("kmers", "batch", "host", "build") else 0
    c["n_seqs"] = 0
    if op in ("seqs", "ranges", "batch", "host", "epoch"):
        c["shape"] = rng.choice(["uniform", "uniform", "lognormal"])
        c["lo"] = rng.choice([1, 20, 31, 100])
        c["hi"] = max(c["lo"], _log(rng, 40, 10_000))
        c["n_seqs"] = max(1, min(_log(rng, 1, 100_000), most, 100_000_000 // c["hi"]))
    if op == "epoch":
        c["epoch_docs"] = max(1, min(_log(rng, 1, 1000), c["docs"]))
    if op == "build":
        c["insert_mode"] = rng.choice([2, 3])
    if op in ("seqs", "ranges", "batch"):
        c["query_path"] = rng.choice([0, 1, 1])
        c["early_exit"] = c["query_path"] == 1 and rng.random() < 0.2
    return c


# ---------------------------------------------------------------- inputs

def _pack(bases):
    """2-bit packed bytes of a flat uint8 tensor whose length is a multiple of 4."""
    q = bases.view(-1, 4)
    return q[:, 0] | (q[:, 1] << 2) | (q[:, 2] << 4) | (q[:, 3] << 6)


def _bases_at(packed, t):
    return (packed[t >> 2] >> (2 * (t & 3)).to(torch.uint8)) & 3


def _corpus(g, n, length):
    """n documents of about `length` bases: packed bytes, CSR offsets (odd starts among them)."""
    L = (length + 3) // 4 * 4
    seeds = torch.randint(0, 4, (max(1, n // 50), L), dtype=torch.uint8, device="cuda", generator=g)
    pick = torch.randint(0, seeds.shape[0], (n,), device="cuda", generator=g)
    packed = torch.zeros(n * L // 4 + 16, dtype=torch.uint8, device="cuda")
    step = max(1, 200_000_000 // L)
    for a in range(0, n, step):
        x = seeds[pick[a:a + step]].view(-1)
        r = torch.randint(0, 1 << 20, x.shape, dtype=torch.int32, device="cuda", generator=g)
        x += (r < (1 << 20) // 100).to(torch.uint8) * (1 + r % 3).to(torch.uint8)  # 1% substitutions
        packed[a * L // 4: a * L // 4 + x.numel() // 4] = _pack(x & 3)
    offs = torch.arange(n + 1, device="cuda") * L
    if n > 1:
        offs[1:n] += torch.randint(0, min(97, L // 4), (n - 1,), device="cuda", generator=g)
    return packed, offs


def _lengths(g, case):
    n, lo, hi = case["n_seqs"], case["lo"], case["hi"]
    if case["shape"] == "lognormal":
        z = torch.randn(n, device="cuda", generator=g, dtype=torch.float64)
        return (300.0 * torch.exp(z)).round().clamp(lo, hi).long()
    return torch.randint(lo, hi + 1, (n,), device="cuda", generator=g)


def _sequences(g, case, corpus, docs, byte_aligned=False):
    """Query sequences, 70% from documents: packed bytes, begins and ends in bases."""
    packed, offs = corpus
    lens = _lengths(g, case)
    n = lens.numel()
    room = (lens + 3) // 4 * 4 if byte_aligned else lens
    begin = torch.cumsum(room, 0) - room
    total = int(room.sum())
    d = torch.randint(0, docs, (n,), device="cuda", generator=g)
    have = offs[d + 1] - offs[d]
    u = torch.rand(n, device="cuda", generator=g, dtype=torch.float64)
    from_doc = (torch.rand(n, device="cuda", generator=g) < 0.7) & (have >= room)
    src = offs[d] + (u * (have - room).clamp(min=0).double()).long()
    out = torch.zeros((total + 3) // 4 * 4, dtype=torch.uint8, device="cuda")
    step = max(1, 50_000_000 // max(1, int(room.max())))
    for a in range(0, n, step):
        b = min(n, a + step)
        r = room[a:b]
        q = torch.repeat_interleave(torch.arange(a, b, device="cuda"), r)
        t0 = int(begin[a])
        t = torch.arange(t0, t0 + q.numel(), device="cuda")
        rnd = torch.randint(0, 1 << 20, t.shape, dtype=torch.int32, device="cuda", generator=g)
        x = _bases_at(packed, torch.where(from_doc[q], src[q] + t - begin[q], 0))
        x = (x + (rnd < (1 << 20) // 1000).to(torch.uint8) * (1 + rnd % 3).to(torch.uint8)) & 3
        out[t0:t0 + q.numel()] = torch.where(from_doc[q], x, (rnd & 3).to(torch.uint8))
    return torch.cat([_pack(out), out.new_zeros(16)]), begin, begin + lens


def _kmers(g, case, corpus, docs):
    """Forward codes of single k-mers, half of them from documents."""
    packed, offs = corpus
    n, k = case["n_kmers"], case["k"]
    d = torch.randint(0, docs, (n,), device="cuda", generator=g)
    u = torch.rand(n, device="cuda", generator=g, dtype=torch.float64)
    start = offs[d] + (u * (offs[d + 1] - offs[d] - k).double()).long()
    present = torch.rand(n, device="cuda", generator=g) < 0.5
    code = torch.zeros(n, dtype=torch.int64, device="cuda")
    for i in range(k):
        x = torch.where(present, _bases_at(packed, start + i).long(),
                        torch.randint(0, 4, (n,), device="cuda", generator=g))
        code = (code << 2) | x
    return code


def _csr(begin, ends):
    return torch.cat([begin, ends[-1:]])


def _pinned(t):
    p = torch.empty(t.shape, dtype=t.dtype, pin_memory=True)
    p.copy_(t)
    return p


def _words(case, seed):
    """Word documents and queries: lists of byte strings from a Zipf-like vocabulary."""
    rng = np.random.default_rng(seed)
    n_vocab = 20_000
    lens = 1 + rng.poisson(6, n_vocab)
    cut = np.concatenate([[0], np.cumsum(lens)])
    letters = rng.integers(97, 123, size=int(cut[-1]), dtype=np.uint8).tobytes()
    vocab = [letters[a:b] for a, b in zip(cut[:-1].tolist(), cut[1:].tolist())]
    cdf = np.cumsum(np.arange(1, n_vocab + 1) ** -1.07)
    terms = np.searchsorted(cdf, rng.random((case["docs"], case["doc_len"])) * cdf[-1])
    docs = [[vocab[t] for t in row] for row in terms.tolist()]
    queries = []
    for _ in range(case["n_seqs"]):
        n = int(rng.integers(case["lo"], case["hi"] + 1))
        if rng.random() < 0.7:  # words of one document
            row = docs[int(rng.integers(0, len(docs)))]
            queries.append([row[i] for i in rng.integers(0, len(row), size=n)])
        else:
            queries.append([vocab[i] for i in rng.integers(0, n_vocab, size=n)])
    return docs, queries


def prepare(case, seed):
    idx = rambo.Index(case["K"], case["B"], case["R"], case["m"], case["eta"], case["k"], seed=7)
    op = case["op"]
    s = {"op": op, "idx": idx}
    if op == "words":
        docs, s["queries"] = _words(case, seed)
        idx.insert_words(np.arange(case["docs"], dtype=np.uint32), docs)
        return s
    knobs = autotune.load_cached(autotune.CACHE_FILE, TUNED[case["tuning"]]) if case["tuning"] else {}
    knobs.update({f: int(case[f]) for f in ("query_path", "early_exit", "insert_mode") if f in case})
    if knobs:
        idx.set_tuning(**knobs)
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    docs = case["docs"]
    corpus = _corpus(g, docs, case["doc_len"])
    ids = torch.arange(docs, dtype=torch.int32, device="cuda")
    if op == "build":  # the pass itself inserts the documents
        s["docs"] = (ids, *corpus)
    else:
        idx.insert_batch_dev(ids, *corpus)
        idx.sync()
        if knobs.get("insert_mode") == 3:  # gives back the buffer that only building needs
            idx.set_tuning(insert_mode=2)
    if op == "epoch":  # documents that arrive now, under the next free ids where there are any
        new = case["epoch_docs"]
        s["docs"] = ((torch.arange(new, device="cuda") + docs).remainder(case["K"]).to(torch.int32),
                     *_corpus(g, new, case["doc_len"]))
    if case["n_kmers"]:
        s["kmers"] = _kmers(g, case, corpus, docs)
    if case["n_seqs"]:
        s["packed"], begin, s["ends"] = _sequences(g, case, corpus, docs, byte_aligned=op == "ranges")
        s["begins"], s["offsets"] = begin, _csr(begin, s["ends"])
    rows = {"out_kmers": case["n_kmers"], "out_seqs": case["n_seqs"]}
    if op == "host":
        s["kmers"] = _pinned(s["kmers"]).numpy().view(np.uint64)
        s["packed"] = _pinned(s["packed"]).numpy()
        s["offsets"] = _pinned(s["offsets"]).numpy().view(np.uint64)
        s.update({f: torch.empty((n, idx.W), dtype=torch.int32, pin_memory=True).numpy()
                  for f, n in rows.items()})
    elif op in ("batch", "ranges"):
        s.update({f: torch.empty((n, idx.W), dtype=torch.int32, device="cuda") for f, n in rows.items()})
    return s


def run(s):
    idx, op = s["idx"], s["op"]
    if op == "words":
        return idx.query_words(s["queries"]).view(np.int32)
    if op == "kmers":
        return idx.query_kmers_dev(s["kmers"])
    if op == "seqs":
        return idx.query_seqs_dev(s["packed"], s["offsets"])
    if op == "ranges":
        return idx.query_ranges_dev(s["packed"], s["begins"], s["ends"], out=s["out_seqs"])
    if op == "batch":
        return idx.query_batch_dev(s["kmers"], s["packed"], s["offsets"], out_kmers=s["out_kmers"],
                                   out_seqs=s["out_seqs"])
    if op == "host":
        idx.query_batch(s["kmers"], s["packed"], s["offsets"], out_kmers=s["out_kmers"],
                        out_seqs=s["out_seqs"])
        return s["out_kmers"], s["out_seqs"]
    idx.insert_batch_dev(*s["docs"])
    if op == "epoch":
        return idx.query_seqs_dev(s["packed"], s["offsets"])
    return idx.query_kmers_dev(s["kmers"])


def work(case):
    """Bytes of one pass: inputs, eta groups of R*B bits per term, answers; for insertion
    the bits of a probe in their sectors, or the index once if that is less.  No
    floating-point arithmetic."""
    row = (case["K"] + 31) // 32 * 4
    group = (case["R"] * case["B"] + 31) // 32 * 4
    probe = case["eta"] * group
    total = case["n_kmers"] * (8 + probe + row)
    if case["op"] == "words":
        terms = case["n_seqs"] * (case["lo"] + case["hi"]) / 2
        return {"bytes": terms * (7 + 8 + probe) + case["n_seqs"] * (8 + row), "flops": 0}
    if case["n_seqs"]:
        if case["shape"] == "lognormal":  # mean of the clipped log-normal lengths, by quadrature
            z = [(i + 0.5) / 100 - 5 for i in range(1000)]
            mean = sum(min(max(300 * math.exp(x), case["lo"]), case["hi"]) * math.exp(-x * x / 2) for x in z)
            mean /= sum(math.exp(-x * x / 2) for x in z)
            terms = max(1.0, mean - case["k"] + 1)
        else:
            lo, hi, k = case["lo"], case["hi"], case["k"]
            mean = (lo + hi) / 2
            terms = sum(max(0, n - k + 1) for n in range(lo, hi + 1)) / (hi - lo + 1)
        total += case["n_seqs"] * (mean / 4 + 8 + terms * probe + row)
    if case["op"] in ("build", "epoch"):
        bases = (case["docs"] if case["op"] == "build" else case["epoch_docs"]) * case["doc_len"]
        touched = min(bases * case["eta"] * min(group, 32 * case["R"]), case["m"] * _group_bytes(case))
        total += bases / 4 + 2 * touched
    return {"bytes": total, "flops": 0}
