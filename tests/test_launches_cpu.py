"""What the library asks of the CUDA runtime, without a GPU: a preloaded fake
runtime (fake_cudart.cpp) writes the calls down instead of running kernels."""
import os
import re
import subprocess
import sys

import pytest

from paper_1910_04358_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))
CUDA = os.path.dirname(os.path.dirname(build._nvcc()))

PRELUDE = """
import ctypes, sys
import numpy as np
from paper_1910_04358_gb300 import rambo
log = ctypes.CDLL(None).fake_cudart_log
log.restype = ctypes.c_char_p
ptr = lambda a: a.ctypes.data
def aligned(nbytes):
    a = np.zeros(nbytes + 256, np.uint8)
    return a[-ptr(a) % 256:][:nbytes]
"""


@pytest.fixture(scope="module")
def calls(tmp_path_factory):
    """calls(code): the lines that the fake runtime wrote while `code` ran."""
    so = str(tmp_path_factory.mktemp("fake") / "fake_cudart.so")
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", f"-I{CUDA}/include", os.path.join(HERE, "fake_cudart.cpp"),
                    "-o", so], check=True)
    build.build()

    def run(code):
        r = subprocess.run([sys.executable, "-c", PRELUDE + code], cwd=os.path.dirname(HERE), text=True,
                           capture_output=True, env=dict(os.environ, LD_PRELOAD=so))
        assert r.returncode == 0, r.stderr
        return r.stdout.splitlines()
    return run


def _stream(line):
    return re.search(r"stream=(\S+)", line).group(1)


def test_set_partition_makes_the_patterns_behind_the_copy(calls):
    lines = calls("""
idx = rambo.Index(100, 32, 4, 256, 2)
log()
idx.set_partition(np.zeros((100, 4), np.uint32))
print(log().decode())
""")
    copy, launch = [l for l in lines if l]
    assert copy.startswith("copy bytes=1600") and "k_patterns" in launch
    assert "stream=" in copy and _stream(copy) == _stream(launch)


def test_shared_memory_limits_do_not_depend_on_the_handle(calls):
    # a kernel's limit outlives the launch: a handle that sets it to its own size
    # lowers it under another thread's launch
    lines = calls("""
from paper_1910_04358_gb300.rambo import load, _check
for K, B, R in [(600, 27, 3), (200, 60, 3), (200, 500, 3), (90, 4000, 3), (300, 31, 4), (100, 32, 4), (60, 1000, 4), (60, 800, 5),
                (60, 650, 5)]:
    idx = rambo.Index(K, B, R, 1 << 12, 2, k=15)
    log()
    idx.set_tuning(insert_mode=3, bin_region_kib=1 + B // 100, early_exit=1)
    ids, offs = np.arange(8, dtype=np.uint32), np.arange(9, dtype=np.uint64) * 100
    idx.insert_batch(ids, np.zeros(300, np.uint8), offs)
    idx.query_kmers(np.arange(50))
    for path in (0, 1, 2):
        idx.set_tuning(query_path=path)
        idx.query_seqs(np.zeros(300, np.uint8), offs)
    print(log().decode())
    idx.close()
""")
    limits, launched = {}, {}
    for line in lines:
        w = line.split()
        if line.startswith("limit "):
            limits.setdefault(w[1], set()).add(int(w[2]))
        elif line.startswith("launch "):
            launched.setdefault(w[1], set()).add(int(re.search(r"smem=(\d+)", line).group(1)))
    for kernel in ("k_answers", "k_insert_bin_apply", "k_insert_bin_scatter", "k_bin_scatter", "k_fused_heavy"):
        assert any(kernel in k for k in limits), kernel
    for kernel, values in limits.items():
        assert len(values) == 1, (kernel, values)
        assert max(values) >= max(launched.get(kernel, {0})) and max(values) <= 227 * 1024, kernel
    assert any(len(v) > 1 for k, v in launched.items() if "k_answers" in k)


def test_sequence_probe_grid_of_a_few_ranges_of_a_large_buffer(calls):
    # blocks for every base of the buffer would nearly all find nothing to do
    lines = calls("""
idx = rambo.Index(100, 100, 5, 256, 2)
L = rambo.load()
z = np.zeros(10, np.uint8)
for n, nbytes in [(500, 1_250_000_000), (5000, 1_250_000_000), (256, 30_080), (20_000, 850_000)]:
    b = np.zeros(n + 1, np.uint64)
    out, ws = np.zeros((n, idx.W), np.uint32), aligned(idx.workspace_bytes("seqs", n))
    log()
    rambo._check(L.rambo_query_ranges_dev(idx._h, n, ptr(z), nbytes, ptr(b), ptr(b) + 8, ptr(out), ptr(ws), ws.size, None), "q")
    print([l for l in log().decode().splitlines() if "k_probe_tiles" in l][0])
""")
    blocks = [int(re.search(r"grid=(\d+),1 ", line).group(1)) for line in lines]
    resident = 152 * 3
    assert resident <= blocks[0] <= 16 * resident and resident <= blocks[1] <= 16 * resident
    assert 120 <= blocks[2] <= 256           # a warp for every 128 k-mers
    assert 2000 <= blocks[3] <= 3500         # about a warp a read


def test_path_1_keeps_the_persistent_launch_for_wide_answers_without_a_byte_table(calls):
    lines = calls("""
L = rambo.load()
z = np.zeros(10, np.uint8)
for K, B, R, tab, n, bases in [(40_000, 250, 8, 1, 3000, 170), (40_000, 250, 8, 1, 2000, 170), (40_000, 250, 6, 1, 3000, 170),
                               (4000, 250, 8, 1, 3000, 170), (5000, 32, 4, 0, 3000, 1000), (5000, 32, 4, 0, 3000, 170),
                               (5000, 32, 4, 1, 3000, 1000)]:
    idx = rambo.Index(K, B, R, 256, 2)
    idx.set_tuning(query_path=1, use_byte_table=tab)
    b = np.zeros(n + 1, np.uint64)
    out, ws = np.zeros((n, idx.W), np.uint32), aligned(idx.workspace_bytes("seqs", n))
    log()
    rambo._check(L.rambo_query_seqs_dev(idx._h, n, ptr(z), n * bases // 4, ptr(b), ptr(out), ptr(ws), ws.size, None), "q")
    print("k_fused" in log().decode())
    idx.close()
""")
    assert lines == ["True", "False", "False", "False", "True", "False", "False"]


def test_word_probe_takes_threads_for_large_batches(calls):
    lines = calls("""
L = rambo.load()
z = np.zeros(10, np.uint8)
for B, n, nbytes in [(32, 1000, 6000), (32, 77_824, 10), (32, 77_825, 10), (32, 1000, 8 * 77_825), (1000, 77_825, 10), (1000, 311_297, 10)]:
    idx = rambo.Index(64, B, 2, 256, 2)
    offs = np.zeros(n + 1, np.uint64)
    out, ws = np.zeros((n, idx.W), np.uint32), aligned(L.rambo_query_words_workspace(idx._h, n))
    log()
    rambo._check(L.rambo_query_words_dev(idx._h, n, ptr(z), nbytes, ptr(offs), ptr(offs), ptr(out), ptr(ws), ws.size, None), "q")
    print("k_probe_words_by_thread" in log().decode())
    idx.close()
""")
    assert lines == ["False", "False", "True", "True", "False", "True"]


def test_sequences_beside_kmer_chunks_of_a_host_call_keep_even_tiles(calls):
    lines = calls("""
idx = rambo.Index(100, 100, 5, 256, 2)
n = 3000
packed, offs = np.zeros(n * 1000 // 4, np.uint8), np.arange(n + 1, dtype=np.uint64) * 1000
for kmers in (np.zeros(0, np.uint64), np.zeros(100, np.uint64)):
    log()
    idx.query_batch(kmers, packed, offs)
    print([l for l in log().decode().splitlines() if "k_probe_tiles" in l][0])
""")
    assert ["Lb1E" in line for line in lines] == [True, False]  # the instance for few items, or not


def test_insertion_grids_of_small_batches(calls):
    # no more blocks than the k-mers that the buffer can hold give work to
    lines = calls("""
idx = rambo.Index(100, 100, 5, 256, 2)
for mode in (2, 3):
    idx.set_tuning(insert_mode=mode)
    for bases in (60, 100_000, 400_000_000):
        if bases > 1_000_000 and mode == 2:
            continue
        L, z, offs = rambo.load(), np.zeros(10, np.uint8), np.zeros(3, np.uint64)
        ids, ws = np.zeros(2, np.uint32), aligned(idx.workspace_bytes("insert", 2))
        log()
        rambo._check(L.rambo_insert_batch_dev(idx._h, 2, ptr(ids), ptr(z), bases // 4, ptr(offs), ptr(ws), ws.size, None), "i")
        print([l for l in log().decode().splitlines() if l.startswith("launch") and "k_insert" in l][0])
""")
    blocks = [int(re.search(r"grid=(\d+),1 ", line).group(1)) for line in lines]
    assert "k_insert_bin_scatter" in lines[2]
    assert blocks == [1, 196, 1, 49, 152 * 3 * 16]
