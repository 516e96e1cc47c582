"""The answer kernels (32 queries at a time) at the edges of their tiles.

Answers are bits, so every comparison with the oracle is for equality.
"""
import numpy as np
import pytest

import oracle
from paper_1910_04358_gb300 import synth

pytestmark = pytest.mark.gpu

# K around the 32-document blocks and 128-document quads; R compiled in (2..6)
# and not (1, 7); tables per warp (up to 2,048 slots) and per block; the
# largest R*B with 16-bit slots and the first past it; eta past one round
GEOMETRIES = [
    # K,   B,     R, eta
    (1, 1, 1, 1),
    (33, 3, 1, 2),
    (128, 20, 2, 2),
    (129, 43, 3, 3),
    (1000, 32, 4, 2),
    (1057, 100, 5, 2),
    (4097, 316, 6, 5),
    (300, 60, 7, 4),
    (500, 700, 3, 2),
    (90, 16383, 1, 2),
    (90, 16384, 1, 2),
]
# repetitions taken four pairs at a time until no query has the documents
MANY_REPETITIONS = [(300, 6, 16, 2), (300, 6, 17, 1), (129, 9, 31, 2), (1000, 20, 128, 3), (70, 40, 200, 5)]


def _dev(torch, a, dt):
    return torch.from_numpy(np.ascontiguousarray(a).view(dt)).cuda()


@pytest.mark.parametrize("K,B,R,eta", GEOMETRIES + MANY_REPETITIONS)
def test_answers_match_oracle(rambo_lib, K, B, R, eta):
    import torch
    p = synth.Params(K=K, B=B, R=R, m=1 << 11, eta=eta, k=15, seed=K)
    rng = np.random.default_rng(K + B)
    corpus = synth.family_corpus(rng, p, n_seeds=max(1, K // 16), doc_len=60, sub_rate=0.02)
    ids = corpus.doc_ids[::2]  # every other document is never inserted
    o = oracle.Rambo(p.K, p.B, p.R, p.m, p.eta, p.k, p.seed)
    idx = rambo_lib.Index(p.K, p.B, p.R, p.m, p.eta, p.k, p.seed)
    packed, offs = synth.pack_many([corpus.doc_bases(int(d)) for d in ids])
    o.insert_batch(ids, packed, offs)
    idx.insert_batch(ids, packed, offs)
    kmers = synth.sample_kmers(rng, corpus, 700, p.k, 0.7)
    want = o.query_kmers(kmers)
    # sequences: the answers come from masks in memory; one shorter than k
    q = synth.sample_queries(rng, corpus, np.concatenate([rng.integers(15, 60, size=69), [7]]), 0.7)
    want_s = o.query_seqs(q.packed, q.offsets)
    dk, dp, do = _dev(torch, kmers, np.int64), _dev(torch, q.packed, np.uint8), _dev(torch, q.offsets, np.int64)
    for n in (1, 31, 32, 33, 700):
        for shift in (0, 1):  # answer rows on and off a 16-byte boundary
            buf = torch.full((n * idx.W + 8,), -1, dtype=torch.int32, device="cuda")
            out = buf[shift:shift + n * idx.W].view(n, idx.W)
            idx.query_kmers_dev(dk[:n], out=out)
            idx.sync()
            assert np.array_equal(rambo_lib.as_u32(out), want[:n]), (n, shift)
            assert (buf[:shift] == -1).all() and (buf[shift + n * idx.W:] == -1).all()
    for ctas in (1, 8):
        idx.set_tuning(expand_ctas_per_sm=ctas)
        got = idx.query_seqs_dev(dp, do)
        idx.sync()
        assert np.array_equal(rambo_lib.as_u32(got), want_s), ctas
    if B % 2 == 0 and idx.info["group_bytes"] <= 512:  # the documents' slots after folding
        idx.fold()
        o.fold()
        assert np.array_equal(idx.query_kmers(kmers), o.query_kmers(kmers))


def test_kmer_answers_latch_bad_codes(rambo_lib):
    idx = rambo_lib.Index(40, 8, 2, 1 << 10, 2, k=15)
    kmers = np.arange(100, dtype=np.uint64)
    kmers[77] = 1 << 31
    with pytest.raises(rambo_lib.RamboError) as e:
        idx.query_kmers(kmers)
    assert e.value.code == rambo_lib.RAMBO_EINVAL
    idx.query_kmers(kmers[:77])


@pytest.mark.parametrize("K,B,R,m,eta", [
    (60, 9, 3, 3001, 1),          # 4-byte groups: one word per record; odd m
    (90, 32, 2, 1 << 12, 3),      # 8-byte groups: one 64-bit word per record
    (200, 31, 4, 1 << 12, 2),     # 16-byte groups: two words per record
    (120, 40, 3, 1 << 12, 5),     # 16-byte groups: a lane per repetition, eta past one pass
    (80, 30, 9, 1 << 11, 2),      # 64-byte groups, nine repetitions
    (50, 3, 40, 1 << 11, 2),      # more repetitions than lanes, groups of few words
    (40, 70, 33, 1 << 10, 1),     # more repetitions than lanes, a lane per repetition
])
def test_insert_record_shapes_match_oracle(rambo_lib, K, B, R, m, eta):
    # documents shorter and longer than a thread's run of k-mers, empty ones
    # among them; direct, binned, and binned with bins that overflow
    p = synth.Params(K=K, B=B, R=R, m=m, eta=eta, k=21, seed=K)
    rng = np.random.default_rng(K * 3 + R)
    lens = np.concatenate([[0, 20, 21, 22, 28, 29, 37], rng.integers(21, 400, size=K - 8), [9001]])
    packed, offs = synth.pack_many([synth.uniform_genome(rng, int(n)) for n in lens])
    ids = rng.permutation(K).astype(np.uint32)
    o = oracle.Rambo(p.K, p.B, p.R, p.m, p.eta, p.k, p.seed)
    o.insert_batch(ids, packed, offs)
    for st in (dict(insert_mode=2), dict(insert_mode=3, bin_region_kib=16),
               dict(insert_mode=3, bin_region_kib=1, insert_bin_records=4096)):
        idx = rambo_lib.Index(p.K, p.B, p.R, p.m, p.eta, p.k, p.seed)
        idx.set_tuning(**st)
        idx.insert_batch(ids, packed, offs)
        words = idx.copy_index().view(np.uint32).reshape(m, -1)
        bits = np.unpackbits(words.view(np.uint8), axis=1, bitorder="little")
        for r in range(R):
            for b in range(B):
                want = np.unpackbits(o.filter_words(r, b).view(np.uint8), bitorder="little")[:m]
                assert np.array_equal(bits[:, r * B + b], want), (st, r, b)
        assert not bits[:, R * B:].any()
        idx.close()


@pytest.mark.parametrize("K,B,R,m,eta", [
    (60, 16, 128, 1 << 12, 2),    # 256-byte groups, the most words a warp sets at once
    (60, 17, 128, 1 << 12, 2),    # 512-byte groups: a lane per repetition
    (60, 20, 128, 4093, 1),
    (50, 9, 256, 1 << 12, 3),     # 512-byte groups, eight repetitions a lane
    (40, 10, 500, 1 << 11, 2),    # groups of two 512-byte chunks
])
def test_insert_records_of_many_repetitions_match_oracle(rambo_lib, K, B, R, m, eta):
    test_insert_record_shapes_match_oracle(rambo_lib, K, B, R, m, eta)


def test_sequence_batches_around_the_prefix_scans(rambo_lib):
    # one block, a cluster of blocks (its shares kept and recounted), three
    # launches; queries of no, one or a few k-mers
    import torch
    p = synth.Params(K=40, B=8, R=2, m=1 << 12, eta=2, k=15, seed=1)
    rng = np.random.default_rng(6)
    corpus = synth.family_corpus(rng, p, n_seeds=8, doc_len=300, sub_rate=0.02)
    n = 131075
    offs = np.concatenate([[0], np.cumsum(rng.integers(12, 20, size=n))]).astype(np.uint64)
    packed = np.concatenate([corpus.packed[:2900]] * (int(offs[-1]) // 11600 + 1) + [np.zeros(16, np.uint8)])
    o = oracle.Rambo(p.K, p.B, p.R, p.m, p.eta, p.k, p.seed)
    o.insert_batch(corpus.doc_ids, corpus.packed, corpus.offsets)
    want = o.query_seqs(packed, offs, threads=4)
    idx = rambo_lib.Index(p.K, p.B, p.R, p.m, p.eta, p.k, p.seed)
    idx.insert_batch(corpus.doc_ids, corpus.packed, corpus.offsets)
    dp, do = _dev(torch, packed, np.uint8), _dev(torch, offs, np.int64)
    for path in (0, 1):
        idx.set_tuning(query_path=path)
        for m in (1, 4095, 4096, 4097, 32768, 32769, 131072, n):
            got = idx.query_seqs_dev(dp, do[:m + 1])
            idx.sync()
            assert np.array_equal(rambo_lib.as_u32(got), want[:m]), (path, m)


@pytest.mark.parametrize("K,B,R,eta", [(300, 32, 4, 2), (300, 60, 3, 3), (200, 100, 5, 1), (64, 400, 6, 2)])
def test_sequence_tiles_match_oracle(rambo_lib, K, B, R, eta):
    # tiles of a query: none, part of one, exactly one and one k-mer more,
    # several; small batches with a fused path set take the same tiles
    import torch
    p = synth.Params(K=K, B=B, R=R, m=(1 << 14) - 3, eta=eta, k=31, seed=2)
    rng = np.random.default_rng(K + R)
    corpus = synth.family_corpus(rng, p, n_seeds=12, doc_len=3000, sub_rate=0.005)
    lens = [0, 30, 31, 62, 63, 94, 157, 158, 159, 286, 287, 1054, 1055, 2500] * 9
    q = synth.sample_queries(rng, corpus, np.array(lens), 0.8)
    o = oracle.Rambo(p.K, p.B, p.R, p.m, p.eta, p.k, p.seed)
    o.insert_batch(corpus.doc_ids, corpus.packed, corpus.offsets)
    want = o.query_seqs(q.packed, q.offsets)
    idx = rambo_lib.Index(p.K, p.B, p.R, p.m, p.eta, p.k, p.seed)
    idx.insert_batch(corpus.doc_ids, corpus.packed, corpus.offsets)
    dp, do = _dev(torch, q.packed, np.uint8), _dev(torch, q.offsets, np.int64)
    for st in (dict(query_path=0), dict(query_path=0, probe_ctas_per_sm=1), dict(query_path=0, probe_min_kmers_per_warp=5000),
               dict(query_path=1, fused_tile_kmers=4096), dict(query_path=1, fused_tile_kmers=1)):
        idx.set_tuning(probe_ctas_per_sm=0, probe_min_kmers_per_warp=0)
        idx.set_tuning(**st)
        got = idx.query_seqs_dev(dp, do)
        idx.sync()
        assert np.array_equal(rambo_lib.as_u32(got), want), st


@pytest.mark.parametrize("path", [0, 1])
def test_overlapping_ranges_have_more_tiles_than_bases(rambo_lib, path):
    # 2,000 ranges over the same 4,000 bases: sixteen times the tiles that the
    # buffer's length suggests
    import torch
    p = synth.Params(K=60, B=16, R=3, m=1 << 14, eta=2, k=31, seed=12)
    rng = np.random.default_rng(9)
    corpus = synth.family_corpus(rng, p, n_seeds=4, doc_len=4000, sub_rate=0.002)
    idx = rambo_lib.Index(p.K, p.B, p.R, p.m, p.eta, p.k, p.seed)
    idx.insert_batch(corpus.doc_ids, corpus.packed, corpus.offsets)
    o = oracle.Rambo(p.K, p.B, p.R, p.m, p.eta, p.k, p.seed)
    o.insert_batch(corpus.doc_ids, corpus.packed, corpus.offsets)
    # most of a document, then bases of none: ranges past it have no answer
    packed = synth.pack_bases(np.concatenate([corpus.doc_bases(0)[:3500], synth.uniform_genome(rng, 500)]))
    begins = rng.integers(0, 100, size=2000)
    ends = rng.integers(3000, 4001, size=2000)
    seqs = [synth.unpack_bases(packed, int(b), int(e - b)) for b, e in zip(begins, ends)]
    qp, qo = synth.pack_many(seqs)
    want = o.query_seqs(qp, qo, threads=4)
    idx.set_tuning(query_path=path)
    got = idx.query_ranges_dev(_dev(torch, packed, np.uint8), _dev(torch, begins.astype(np.int64), np.int64),
                               _dev(torch, ends.astype(np.int64), np.int64))
    idx.sync()
    assert np.array_equal(rambo_lib.as_u32(got), want)
    assert 0 < want.any(axis=1).sum() < 2000


def _all_paths_match(rambo_lib, torch, idx, o, kmers, q):
    dk, dp, do = _dev(torch, kmers, np.int64), _dev(torch, q.packed, np.uint8), _dev(torch, q.offsets, np.int64)
    want, want_k = o.query_seqs(q.packed, q.offsets), o.query_kmers(kmers)
    # (early exit keeps a batch of any size on the persistent launch)
    for st in (dict(query_path=0), dict(query_path=1, early_exit=1), dict(query_path=2, early_exit=0), dict(query_path=3)):
        idx.set_tuning(**st)
        got, got_k = idx.query_seqs_dev(dp, do), idx.query_kmers_dev(dk)
        idx.sync()
        assert np.array_equal(rambo_lib.as_u32(got), want), st
        assert np.array_equal(rambo_lib.as_u32(got_k), want_k), st
    return want


@pytest.mark.parametrize("K,B,R", [(120, 16, 3), (300, 60, 4), (70, 8, 8)])
def test_fold_of_an_explicit_partition(rambo_lib, K, B, R):
    import torch
    p = synth.Params(K=K, B=B, R=R, m=1 << 12, eta=2, k=21, seed=9)
    rng = np.random.default_rng(K * B + R)
    corpus = synth.family_corpus(rng, p, n_seeds=max(1, K // 12), doc_len=200, sub_rate=0.02)
    q = synth.sample_queries(rng, corpus, rng.integers(15, 150, size=150), 0.8)
    kmers = synth.sample_kmers(rng, corpus, 300, p.k, 0.8)
    phi = rng.integers(0, B, size=(K, R)).astype(np.uint32)
    o = oracle.Rambo(p.K, p.B, p.R, p.m, p.eta, p.k, p.seed)
    idx = rambo_lib.Index(p.K, p.B, p.R, p.m, p.eta, p.k, p.seed)
    for x in (o, idx):
        x.set_partition(phi)

    def insert(ids):
        packed, offs = synth.pack_many([corpus.doc_bases(int(d)) for d in ids])
        for x in (o, idx):
            x.insert_batch(np.asarray(ids, dtype=np.uint32), packed, offs)

    insert(corpus.doc_ids[::2])
    for fold in (False, True, True):
        if fold:
            idx.fold()
            o.fold()
        assert _all_paths_match(rambo_lib, torch, idx, o, kmers, q).any()
        assert np.array_equal(idx.partition(), phi % idx.B)
        if fold:  # documents that are there already and new ones, after the fold
            insert(corpus.doc_ids[:K // 2])
            _all_paths_match(rambo_lib, torch, idx, o, kmers, q)


def test_insertion_right_after_set_partition_uses_the_new_map(rambo_lib):
    # the last documents of a map that takes a while to copy, inserted with one
    # k-mer each: the only group that is set holds the new buckets and no other
    K, B, R = 1 << 20, 32, 4
    rng = np.random.default_rng(3)
    packed, offs = synth.pack_many([synth.uniform_genome(rng, 15)] * 64)
    ids = np.arange(K - 64, K, dtype=np.uint32)
    for i in range(20):
        phi = rng.integers(0, B, size=(K, R)).astype(np.uint32)
        with rambo_lib.Index(K, B, R, 1 << 8, 1, 15, seed=i) as idx:
            idx.set_partition(phi)
            idx.insert_batch(ids, packed, offs)
            rows = idx.copy_index().reshape(1 << 8, -1)
        hit = np.nonzero(rows.any(axis=1))[0]
        assert hit.size == 1, i
        got = np.nonzero(np.unpackbits(rows[hit[0]], bitorder="little"))[0]
        assert np.array_equal(got, np.unique(phi[ids] + B * np.arange(R, dtype=np.uint32))), i


@pytest.mark.parametrize("B,R", [(10, 3), (32, 4), (60, 4), (100, 5), (200, 5), (400, 6), (500, 8), (600, 8)])
def test_few_items_in_a_large_buffer(rambo_lib, B, R):
    # fewer items than resident warps over bases for 512 k-mers a warp and more:
    # tiles of 128 k-mers, a query's tiles of one warp in one mask.  A few ranges
    # of the buffer, items that cover it (of some tiles, and of thousands), and
    # the same with a fixed grid, whose warps take many tiles.
    import torch
    p = synth.Params(K=70, B=B, R=R, m=(1 << 14) + 5, eta=2, k=31, seed=5)
    rng = np.random.default_rng(B)
    corpus = synth.family_corpus(rng, p, n_seeds=6, doc_len=4000, sub_rate=0.001)
    o = oracle.Rambo(p.K, p.B, p.R, p.m, p.eta, p.k, p.seed)
    idx = rambo_lib.Index(p.K, p.B, p.R, p.m, p.eta, p.k, p.seed)
    for x in (o, idx):
        x.insert_batch(corpus.doc_ids, corpus.packed, corpus.offsets)
    total = 152 * 24 * 512 + 4001
    bases = synth.uniform_genome(rng, total)
    at = np.arange(0, total - 4100, 6000)
    for i, a in enumerate(at):  # documents here and there, random bases between
        bases[a:a + 4000] = corpus.doc_bases(i % p.K)
    packed = synth.pack_bases(bases)
    few = np.sort(rng.choice(at, 40, replace=False))
    cases = [(few, few + rng.choice([20, 31, 157, 158, 159, 1000, 4000], size=40)),
             (np.arange(0, total, 2500), np.append(np.arange(2500, total, 2500), total)),
             (np.array([0, 9, 1000]), np.array([9, 1000, total]))]
    dp = _dev(torch, np.concatenate([packed, np.zeros(16, np.uint8)]), np.uint8)
    hits = 0
    for begins, ends in cases:
        qp, qo = synth.pack_many([bases[b:e] for b, e in zip(begins, ends)])
        want = o.query_seqs(qp, qo, threads=4)
        hits += np.count_nonzero(want)
        for ctas in (0, 1):
            idx.set_tuning(query_path=0, probe_ctas_per_sm=ctas)
            got = idx.query_ranges_dev(dp, _dev(torch, begins.astype(np.int64), np.int64),
                                       _dev(torch, ends.astype(np.int64), np.int64))
            idx.sync()
            assert np.array_equal(rambo_lib.as_u32(got), want), (len(begins), ctas)
    assert hits > 40


@pytest.mark.parametrize("K,B,R,eta", [
    (60, 9, 3, 2), (60, 20, 3, 1), (60, 32, 4, 3),   # 4-, 8- and 16-byte groups: 2, 2 and 4 lanes a term
    (60, 60, 4, 9), (60, 100, 5, 2),                 # 32 bytes and nine seeds: 16; 64 bytes: 4
    (60, 1000, 2, 2), (40, 1000, 5, 33),             # 256 bytes: 16; two 512-byte chunks, more seeds than lanes
])
def test_word_queries_around_a_warp_per_term(rambo_lib, K, B, R, eta):
    # 152 SMs x 64 warps: up to 9,728 terms have a warp each, more share it, and
    # from 77,825 queries on (groups of 256 bytes: 311,297) a term is a thread's
    rng = np.random.default_rng(B + eta)
    vocab = synth.word_vocabulary(rng, 900)
    docs = synth.word_corpus(rng, K, vocab, 60)
    o = oracle.Rambo(K, B, R, 5003, eta, seed=5)
    idx = rambo_lib.Index(K, B, R, 5003, eta, seed=5)
    for d in range(K):
        o.insert_words(d, [vocab[i] for i in docs[d]])
    idx.insert_words(np.arange(K), [[vocab[i] for i in docs[d]] for d in range(K)])
    # queries of a document's words, of words of none, of no word, and with empty words
    pool = [[vocab[j] for j in rng.choice(docs[int(rng.integers(0, K))], size=int(s))] for s in rng.integers(1, 5, size=60)]
    pool += [[], [b""], [b"", vocab[int(docs[0][0])]], [b"none of them"]]
    want_of = [o.query_words(q) for q in pool]
    assert np.count_nonzero(want_of) > 30
    for terms in (1, 9727, 9728, 9729, 20_011, 800_000 if B == 1000 else 300_000):
        pick, t = [], 0
        while t < terms:
            i = int(rng.integers(0, len(pool)))
            if t + len(pool[i]) <= terms:
                pick.append(i)
                t += len(pool[i])
        got = idx.query_words([pool[i] for i in pick])
        assert np.array_equal(got, np.stack([want_of[i] for i in pick])), terms


def test_word_answers_that_are_held_are_not_page_locked(rambo_lib):
    import torch
    idx = rambo_lib.Index(300, 20, 3, 5003, 2)
    docs = [[b"w%d" % i, b"all"] for i in range(300)]
    idx.insert_words(np.arange(300), docs)
    pinned = lambda a: torch.from_numpy(a.view(np.int32)).is_pinned()
    held = [idx.query_words([[b"w%d" % i], [b"all"]]) for i in range(20)]
    assert sum(pinned(a) for a in held) == 2
    parts = [a[1:] for a in held[:2]]  # views keep the whole blocks
    held = [a.copy() for a in held]
    later = [idx.query_words([[b"w%d" % i], [b"all"]]) for i in range(20)]
    assert not any(pinned(a) for a in later)
    for i, (a, b) in enumerate(zip(held, later)):
        assert np.array_equal(a, b) and i in rambo_lib.answer_docs(a[0]) and rambo_lib.answer_docs(a[1]).size == 300
    assert all(rambo_lib.answer_docs(p[0]).size == 300 for p in parts)
    del parts
    for _ in range(5):  # the last answers go when the next ones come: no copy
        last = idx.query_words([[b"all"]])
        assert pinned(last) and rambo_lib.answer_docs(last[0]).size == 300


def test_words_on_any_stream(rambo_lib):
    # a stream is whatever has its handle, as for every other call
    import types

    import torch
    idx = rambo_lib.Index(30, 10, 3, 5003, 2)
    side = torch.cuda.Stream()
    for i, stream in enumerate((None, side, torch.cuda.ExternalStream(side.cuda_stream),
                                types.SimpleNamespace(cuda_stream=side.cuda_stream))):
        idx.insert_words([i], [[b"word%d" % i]], stream=stream)
        got = idx.query_words([[b"word%d" % i], []], stream=stream)
        assert i in rambo_lib.answer_docs(got[0]) and rambo_lib.answer_docs(got[1]).size == i + 1


@pytest.mark.parametrize("K,B,R,eta", [
    (50, 9, 3, 2),       # 4-byte groups
    (200, 31, 4, 1),     # 16 bytes, patterns in shared memory
    (3000, 31, 4, 2),    # ... and too many documents for it
    (120, 100, 5, 3),    # 64 bytes, a lane per repetition
])
def test_binned_insertion_around_its_small_batches(rambo_lib, K, B, R, eta):
    # batches of few k-mers are applied in smaller units, from 5 units of 2,048
    # records an SM on in full ones; few and many documents, one of them long
    import torch
    edge = 152 * 5 * 2048 // eta
    rng = np.random.default_rng(K)
    packed = torch.from_numpy(rng.integers(0, 256, size=edge // 2 + 64, dtype=np.uint8)).cuda()
    for bases in (31, 5000, 60_000, edge - 8, edge + 8, 2 * edge):
        cuts = np.sort(rng.integers(0, bases + 1, size=min(K, bases // 200 + 1) - 1))
        offs = torch.from_numpy(np.concatenate([[0], cuts, [bases]]).astype(np.int64)).cuda()
        ids = torch.from_numpy(rng.permutation(K)[:offs.numel() - 1].astype(np.int32)).cuda()
        got = []
        for st in (dict(insert_mode=2), dict(insert_mode=3, bin_region_kib=64), dict(insert_mode=3, bin_region_kib=512)):
            with rambo_lib.Index(K, B, R, 1 << 15, eta, 31, 3) as idx:
                idx.set_tuning(**st)
                idx.insert_batch_dev(ids, packed[:(bases + 3) // 4], offs)
                idx.sync()
                got.append(idx.copy_index())
        assert got[0].any() and np.array_equal(got[0], got[1]) and np.array_equal(got[0], got[2]), bases
