"""The library's host code without a GPU: a stand-in for the CUDA runtime (fake_cudart.c, preloaded into a process of
its own) records what each call allocates, clears, copies and launches, and runs no kernel."""
import os
import re
import shutil
import subprocess
import sys

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)

SETUP = r"""
import ctypes as C, math, sys
from types import SimpleNamespace
sys.path.insert(0, sys.argv[1])
from paper_2511_21647_gb300 import _lib as L, rca as R
def geometry(n_el=32, nz=80, ns=256, P=8, K=1, us=2):
    return SimpleNamespace(n_el=n_el, P=P, K=K, nz=nz, ns=ns, us=us, pitch=0.2e-3, fc=7.8e6, fs=31.2e6, c=1540.0,
                           z0=5e-3, dz=0.1e-3, fnum=1.0, ang_rc=[0.05] * K, ang_cr=[-0.05] * K)
keep = []
def buf(n):
    b = C.create_string_buffer(n + 64)
    keep.append(b)
    return (C.addressof(b) + 63) // 64 * 64
def mark(s):
    R.rca_fp32_probe(h, 0, 1, buf(64))     # a launch of k_fp32_probe in the record
h = R.rca_create(0)
"""


@pytest.fixture(scope="module")
def runtime(tmp_path_factory):
    if not shutil.which("gcc"):
        pytest.skip("needs gcc")
    from paper_2511_21647_gb300 import build
    build()
    so = str(tmp_path_factory.mktemp("fake") / "libfake_cudart.so")
    subprocess.run(["gcc", "-shared", "-fPIC", "-O1", "-I/usr/local/cuda/include", os.path.join(HERE, "fake_cudart.c"), "-o", so],
                   check=True)
    return so


def record(runtime, tmp_path, script, args=""):
    """the log of `script`, as lists of words"""
    log = str(tmp_path / "log.txt")
    env = dict(os.environ, LD_PRELOAD=runtime, FAKE_CUDART_LOG=log, FAKE_CUDART_ARGS=args)
    r = subprocess.run([sys.executable, "-c", SETUP + script, ROOT], env=env, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-3000:]
    return [line.split() for line in open(log)]


def launch(log, kernel):
    return next(i for i, w in enumerate(log) if w[0] == "launch" and kernel in w[1])


def int32(word):
    return int(word) & 0xffffffff


@pytest.mark.parametrize("call", ["detect2d", "detect_map"])
def test_candidate_counts_are_cleared_before_detection(runtime, tmp_path, call):
    """a detection block that gives up writes no count: its slots have to be empty, not what an earlier call left"""
    script = r"""
g = R.rca_geometry_create(h, geometry())
t = R.rca_delay_tables(h, g)
A, M, out, n = buf(4 * 2 * 4 * 80 * 32 * 4), buf(64), buf(40 * 64), buf(64)
mark("call")
""" + (r"""
R.ulm_detect2d(h, t, A, M, 4, R.make_ulm_params(), out, 64, n)
""" if call == "detect2d" else r"""
R.ulm_detect_map(h, t, buf(4 * 2 * 4 * 80 * 32 * 4 * 16), 4, A, M, 4, 0.5, 0.1, out, 64, n)
""")
    log = record(runtime, tmp_path, script, "k_gather:5")
    begin, det = launch(log, "k_fp32_probe"), launch(log, "k_detect")
    gather = log[launch(log, "k_gather")]
    cnt, part, total, nslots = int(gather[6]), int(gather[7]), int(gather[8]), int32(gather[9])
    assert nslots == 4 * 2 * 4 * (3 if call == "detect2d" else 11)

    def cleared(p, n):
        return any(w[0] == "memset" and int(w[1]) <= p and p + n <= int(w[1]) + int(w[2]) for w in log[begin:det])

    assert cleared(total, 8) and cleared(part, 4 * ((nslots + 255) // 256))
    assert cleared(cnt, 4 * nslots)


def test_reserved_workspace_serves_the_detection(runtime, tmp_path):
    """after rca_reserve the detection allocates nothing (a capture would refuse it)"""
    log = record(runtime, tmp_path, r"""
for nz, F in ((80, 4), (31, 1), (250, 16)):
    geo = geometry(nz=nz, ns=1100)
    g = R.rca_geometry_create(h, geo)
    t = R.rca_delay_tables(h, g)
    A, M, out, n = buf(F * 2 * 4 * nz * 32 * 4), buf(64), buf(40 * 64), buf(64)
    R.rca_reserve(h, g, F)
    mark("call")
    R.ulm_detect2d(h, t, A, M, F, R.make_ulm_params(), out, 64, n)
    mark("end")
""")
    marks = [i for i, w in enumerate(log) if w[0] == "launch" and "k_fp32_probe" in w[1]]
    assert len(marks) == 6
    for a, b in zip(marks[::2], marks[1::2]):
        assert [w for w in log[a:b] if w[0] == "launch" and "k_gather" in w[1]]
        assert not [w for w in log[a:b] if w[0] == "malloc"]


def test_inference_over_its_input_goes_through_the_own_heatmap(runtime, tmp_path):
    """a heatmap over the memory of the input planes or of their maxima is not stored while others are read"""
    log = record(runtime, tmp_path, r"""
B, H, W = 6, 20, 32
px = B * H * W
net = R.ulm_cnn_create(h, max_pixels=px)
mem = buf(4 * 40 * px)
ends = 4 * 16 * px
for A, M, heat in ((mem, 0, mem), (mem + 64, 0, mem), (mem + ends - 4, 0, mem), (mem, 0, mem + 4 * px - 16), (mem + ends, mem + 64, mem),
                   (mem + ends + 64, mem + ends - 4, mem),
                   (mem + ends, 0, mem), (mem, 0, mem + 4 * px), (mem + ends, mem + ends + 4 * px, mem), (mem, mem + 4 * px, mem + 4 * px + 16)):
    mark("call")
    R.ulm_cnn_infer(net, A, M or None, 2, B, H, W, heat)
mark("end")
""")
    marks = [i for i, w in enumerate(log) if w[0] == "launch" and "k_fp32_probe" in w[1]]
    copied = [any(w[0] == "memcpy" for w in log[a:b]) for a, b in zip(marks, marks[1:])]
    assert copied == [True] * 6 + [False] * 4


def test_iteration_asks_for_the_shared_memory_it_uses(runtime, tmp_path):
    """the subspace iteration's basis and products, and C's rows only for the kernels that keep them there"""
    sizes = [(9, 3), (300, 16), (320, 32), (321, 16), (360, 30), (400, 4), (512, 16), (512, 22)]
    log = record(runtime, tmp_path, rf"""
g = R.rca_geometry_create(h, geometry(nz=4))
t = R.rca_delay_tables(h, g)
for F, rank in {sizes}:
    R.rca_clutter_svd(h, t, buf(F * 2 * 7 * 32 * 8), F, rank)
""")
    found = [w for w in log if w[0] == "launch" and "k_svd_iterate" in w[1]]
    assert len(found) == len(sizes)
    for (F, rank), w in zip(sizes, found):
        nb, rows, in_smem = rank + 1, -(-F // 8), "Lb1E" in w[1]
        assert int(w[4]) == 8 * (F * (nb | 1) + rows * nb + (rows * (F | 1) if in_smem else 0)), (F, rank)
        assert in_smem == (F <= 320) and int(w[4]) <= 227 * 1024 - 1024


@pytest.mark.parametrize("widths,form", [((32,), (1, 2)), ((32, 32), (1, 2)), ((32, 64), (4, 0)), ((36,), (4, 0)), ((64,), (4, 0)),
                                         ((96,), (8, 0)), ((96, 32), (8, 0)), ((128, 32), (8, 0))])
def test_batch_row_loop_fits_its_tiles(runtime, tmp_path, widths, form):
    """rows per thread and pixel pairing of the batch kernel: the exact split form only where every ensemble's tiles have
    whole runs for it, else the loop with the tallest ensemble's rows per thread (tiles of 16 rows)"""
    log = record(runtime, tmp_path, rf"""
items = []
for n_el in {widths}:
    g = R.rca_geometry_create(h, geometry(n_el=n_el, P=4))
    t = R.rca_delay_tables(h, g)
    items.append(dict(tables=t, rf=buf(3 * 2 * n_el * 256 * 4), n_frames=3, planes=buf(3 * 4 * n_el // 4 * 80 * n_el * 8)))
b = R.rca_batch_create(h, items, L.RCA_F32, L.RCA_C32, L.RCA_C32)
R.rca_batch_set_mode(b, L.RCA_BATCH_STAGED)
R.rca_batch_run(b, False, h)
""")
    names = [w[1] for w in log if w[0] == "launch" and "k_batch" in w[1]]
    assert len(names) == 4
    for name in names:
        maxr, _, _, pair = (int(x) for x in re.findall(r"Li(\d+)E", name))
        assert (maxr, pair) == form


def test_gather_spreads_few_chunks_of_slots(runtime, tmp_path):
    """chunks of 256 candidate slots: up to eight blocks each while they are few, one for a long ensemble"""
    log = record(runtime, tmp_path, r"""
g = R.rca_geometry_create(h, geometry())
t = R.rca_delay_tables(h, g)
out, n = buf(40 * 64), buf(64)
for F in (1, 64, 300, 1700, 3000):
    R.ulm_detect2d(h, t, buf(64), buf(64), F, R.make_ulm_params(), out, 64, n)
""")
    grids = [tuple(int(x) for x in w[2].split(",")) for w in log if w[0] == "launch" and "k_gather" in w[1]]
    assert grids == [(1, 8, 1), (6, 8, 1), (29, 8, 1), (160, 3, 1), (282, 2, 1)]
