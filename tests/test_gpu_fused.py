"""The persistent sequence query (path 1) where the library takes it: batches
above its smallest, groups wider than a lane, and one-lane groups beside the
k-mer chunks of a host call.  Every case asserts from the profile's launch
counts that the persistent launch ran.  Answers are bits: all comparisons are
for equality with the oracle.
"""
import numpy as np
import pytest

import oracle
from paper_1910_04358_gb300 import synth

pytestmark = pytest.mark.gpu

# a batch of SMs x 24 x fused_tile_kmers bases and more takes the persistent launch
BASES = 152 * 24 * 64 + 4000


def _dev(torch, a, dt):
    return torch.from_numpy(np.ascontiguousarray(a).view(dt)).cuda()


def _case(rambo_lib, K, B, R, eta, lengths, m=(1 << 14) - 3, doc_len=700):
    p = synth.Params(K=K, B=B, R=R, m=m, eta=eta, k=31, seed=K)
    rng = np.random.default_rng(K + B * R + eta)
    corpus = synth.family_corpus(rng, p, n_seeds=max(4, K // 40), doc_len=doc_len, sub_rate=0.01)
    q = synth.sample_queries(rng, corpus, np.asarray(lengths), 0.7)
    o = oracle.Rambo(p.K, p.B, p.R, p.m, p.eta, p.k, p.seed)
    idx = rambo_lib.Index(p.K, p.B, p.R, p.m, p.eta, p.k, p.seed)
    for x in (o, idx):
        x.insert_batch(corpus.doc_ids, corpus.packed, corpus.offsets)
    return rng, corpus, q, o, idx


def _persistent(idx, call):
    """The call's result; it took the persistent launch (counted with its
    preparation and its heavy pass as three) and no expansion of its own."""
    idx.profile_reset()
    out = call()
    n = {k: v["launches"] for k, v in idx.profile_read().items()}
    assert n["probe_seqs"] == 3 and n["expand"] == 0, n
    return out


@pytest.mark.parametrize("K,B,R,eta", [
    (300, 60, 4, 2),     # 32-byte groups, two lanes each
    (300, 100, 5, 1),    # 64 bytes
    (300, 100, 5, 3),
    (2100, 100, 5, 2),   # answers past 64 words
    (200, 200, 5, 2),    # 128 bytes
    (120, 400, 5, 4),    # 256 bytes
    (90, 500, 8, 2),     # 512 bytes
    (90, 500, 8, 5),
])
def test_persistent_launch_matches_oracle(rambo_lib, K, B, R, eta):
    import torch
    lengths = np.concatenate([[0, 30, 31, 62, 63, 94, 95, 158, 159, 700], np.random.default_rng(1).integers(0, 420, size=1150)])
    rng, corpus, q, o, idx = _case(rambo_lib, K, B, R, eta, lengths)
    assert BASES < 4 * q.packed.size
    want = o.query_seqs(q.packed, q.offsets, threads=4)
    dp, do = _dev(torch, q.packed, np.uint8), _dev(torch, q.offsets, np.int64)
    for st in (dict(fused_tile_kmers=64, fused_short_max=40), dict(fused_tile_kmers=64, fused_short_max=1 << 20),
               dict(fused_tile_kmers=32, fused_short_max=0, probe_ctas_per_sm=1),
               dict(fused_tile_kmers=1, fused_short_max=300, use_byte_table=0),
               dict(fused_tile_kmers=64, fused_short_max=50, fused_async=1)):
        idx.set_tuning(query_path=1, **st)
        got = _persistent(idx, lambda: idx.query_seqs_dev(dp, do))
        idx.sync()
        assert np.array_equal(rambo_lib.as_u32(got), want), st


@pytest.mark.parametrize("K", [2100, 5000])
def test_persistent_launch_with_answers_of_several_chunks(rambo_lib, K):
    # long queries keep a few passing buckets, single k-mers dozens, sequences
    # shorter than k all 1,896: with the byte table, and without it through the
    # decoded list or, past 32 buckets, the heavy pass (answers of several chunks)
    import torch
    lengths = np.concatenate([np.random.default_rng(2).integers(31, 400, size=1150), np.full(40, 31), np.full(5, 10)])
    rng, corpus, q, o, idx = _case(rambo_lib, K, 316, 6, 2, lengths, m=1 << 15, doc_len=500)
    assert BASES < 4 * q.packed.size
    want = o.query_seqs(q.packed, q.offsets, threads=4)
    pops = np.unpackbits(want.view(np.uint8), axis=1).sum(axis=1)
    assert (pops[-5:] == K).all() and (pops[:1150] < K).all()
    dp, do = _dev(torch, q.packed, np.uint8), _dev(torch, q.offsets, np.int64)
    for st in (dict(use_byte_table=1), dict(use_byte_table=0)):
        for shape in (dict(fused_tile_kmers=64, fused_short_max=40), dict(fused_tile_kmers=64, fused_short_max=1024),
                      dict(fused_tile_kmers=1, fused_short_max=0)):
            idx.set_tuning(query_path=1, byte_table_max_mb=64, **st, **shape)
            got = _persistent(idx, lambda: idx.query_seqs_dev(dp, do))
            idx.sync()
            assert np.array_equal(rambo_lib.as_u32(got), want), (st, shape)


@pytest.mark.parametrize("K,B,R,eta", [
    (600, 10, 3, 2),     # 4-byte groups
    (600, 20, 3, 1),     # 8 bytes
    (600, 32, 4, 2),     # 16 bytes
    (600, 32, 4, 1),
    (600, 32, 4, 3),
    (2100, 32, 4, 2),    # answers past 64 words
])
def test_persistent_launch_beside_kmer_chunks_of_a_host_call(rambo_lib, K, B, R, eta):
    # one-lane groups: the gathers through registers or staged in shared memory
    import torch
    lengths = np.concatenate([[0, 30, 31, 62, 700], np.random.default_rng(3).integers(0, 420, size=1150)])
    rng, corpus, q, o, idx = _case(rambo_lib, K, B, R, eta, lengths, m=1 << 15)
    assert BASES < 4 * q.packed.size
    kmers = synth.sample_kmers(rng, corpus, 3001, 31, 0.5)
    want, want_k = o.query_seqs(q.packed, q.offsets, threads=4), o.query_kmers(kmers, threads=4)
    pin = [torch.zeros(w.shape, dtype=torch.int32).pin_memory().numpy() for w in (want_k, want)]
    for st in (dict(fused_async=1, fused_tile_kmers=64, fused_short_max=1024),
               dict(fused_async=1, fused_tile_kmers=64, fused_short_max=40),
               dict(fused_async=1, fused_tile_kmers=1, fused_short_max=0, host_fused_ctas_per_sm=3),
               dict(fused_async=0, fused_tile_kmers=64, fused_short_max=40, branch_priority=1),
               dict(fused_async=0, fused_tile_kmers=64, fused_short_max=0, probe_ctas_per_sm=2, branch_priority=2)):
        idx.set_tuning(query_path=1, host_fused_ctas_per_sm=1)
        idx.set_tuning(host_chunk_kmers=1000, host_slots=4, host_direct=1, **st)
        for out in (pin, [None, None]):  # answers straight into page-locked memory, or staged
            got_k, got = _persistent(idx, lambda: idx.query_batch(kmers, q.packed, q.offsets, *out))
            assert np.array_equal(got_k, want_k) and np.array_equal(got, want), st
            if out[0] is not None:
                for a in out:
                    a[:] = 0


@pytest.mark.parametrize("use_byte_table", [0, 1])
@pytest.mark.parametrize("K", [90, 1025, 2049, 4097, 8200])  # one, two, four and eight words a lane, and more
def test_expansion_of_groups_past_the_slot_tables(rambo_lib, K, use_byte_table):
    # R * B of 16,384 and more: answers row by row, or through the byte table
    rng, corpus, q, o, idx = _case(rambo_lib, K, 4100, 4, 2, [0, 30, 31, 40, 90, 200] * 20, m=1 << 11, doc_len=80)
    kmers = synth.sample_kmers(rng, corpus, 200, 31, 0.7)
    idx.set_tuning(use_byte_table=use_byte_table, byte_table_max_mb=4096)
    assert np.array_equal(idx.query_seqs(q.packed, q.offsets), o.query_seqs(q.packed, q.offsets))
    assert np.array_equal(idx.query_kmers(kmers), o.query_kmers(kmers))
