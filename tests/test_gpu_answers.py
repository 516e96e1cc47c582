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


def _dev(torch, a, dt):
    return torch.from_numpy(np.ascontiguousarray(a).view(dt)).cuda()


@pytest.mark.parametrize("K,B,R,eta", GEOMETRIES)
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
