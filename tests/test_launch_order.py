"""Host code of the library without a GPU, above all the order of an iteration's
kernels: its object files linked against tests/_fakecuda.cpp, which records every launch with the
launches that streams and events put before it.  Kernels that share memory must
be ordered on every annihilation path, for a single run and for a batch:

  split -> attempt     the bucket split clears the counter (DevState::nspawn)
                       whose value the spawning takes as a staging slot
  split -> bucket      splitter keys, bucket counts
  det_pass -> attempt  attempt offsets, flags
  attempt -> bucket / match   the staged spawns
"""
from __future__ import annotations

import ctypes as C
import os
import re
import shutil
import subprocess

import pytest

from paper_1811_11679_gb300 import build, hande, inputs
from test_gpu_tc_gemm_paths import SHAPES

HERE = os.path.dirname(os.path.abspath(__file__))
BUCKETS = [("det_pass", "attempt"), ("split", "attempt"), ("split", "bucket"), ("attempt", "bucket"),
           ("bucket", "scatter")]
HASH = [("det_pass", "attempt"), ("attempt", "match"), ("match", "decide"), ("decide", "place"), ("place", "write")]


@pytest.fixture(scope="module")
def recorder(tmp_path_factory):
    objs = [os.path.join(build.OUT, u.replace(".cu", ".o")) for u in build.UNITS]
    build.build(force=not all(os.path.exists(o) for o in objs))
    toolkit = os.path.dirname(os.path.dirname(os.path.realpath(build.nvcc())))
    include = next(p for p in (os.path.join(toolkit, "include"), "/usr/local/cuda/include") if os.path.isdir(p))
    so = str(tmp_path_factory.mktemp("fake") / "libhande_recorded.so")
    # -Bsymbolic: the library's CUDA calls bind to the definitions linked here
    subprocess.run([shutil.which("g++") or "c++", "-std=c++17", "-O1", "-shared", "-fPIC", "-Wl,-Bsymbolic",
                    "-I", include, os.path.join(HERE, "_fakecuda.cpp"), *objs, "-o", so], check=True)
    mp = pytest.MonkeyPatch()
    mp.setattr(hande, "_lib", None)
    mp.setattr(hande._build, "LIB", so)
    lib = hande.load(build_if_needed=False)
    lib.fake_name.restype = C.c_char_p
    yield lib
    mp.undo()


def _launches(lib):
    """(kernel, its index), the kernels' names without prefixes and template arguments."""
    out = []
    for i in range(lib.fake_count()):
        m = re.search(r"kb?_([a-z_]*[a-z])(?=I[A-Z]|E[A-Zv])", lib.fake_name(i).decode())
        out.append((m.group(1) if m else "", i))
    return out


def _check_orders(lib, pairs):
    seen = _launches(lib)
    for first, then in pairs:
        a = [i for n, i in seen if n == first]
        b = [i for n, i in seen if n == then]
        assert a and len(a) == len(b), (first, then, seen)
        for x, y in zip(a, b):   # the same iteration of the same group
            assert lib.fake_before(x, y), f"{then} does not wait for {first}"


def _run(annihilation, seed=7, norb=38):
    s = inputs.ueg_system(14, norb, 1.0)
    return s, inputs.qmc_params(tau=0.002, target_population=5000, initiator=1, real_amplitudes=1, spawn_cutoff=0.1,
                                init_pop=100, seed=seed, annihilation=annihilation, state_capacity=20000,
                                spawn_capacity=40000)


@pytest.mark.parametrize("annihilation", [0, 1, 2])
@pytest.mark.parametrize("n", [1, 9])            # one iteration, and the graphs of four
def test_single_run(recorder, annihilation, n):
    g = hande.Hande(*_run(annihilation), stream=1, torch_memory=False)
    recorder.fake_reset()
    g.iterate(n)
    _check_orders(recorder, BUCKETS if annihilation else HASH)
    g.close()


@pytest.mark.parametrize("annihilation", [0, 1, 2])
def test_batch(recorder, annihilation):
    runs = [_run(annihilation, seed) for seed in (1, 2)] + [_run(annihilation, 3, norb=19)]
    b = hande.HandeBatch([s for s, _ in runs], [q for _, q in runs], stream=1, torch_memory=False)
    recorder.fake_reset()
    b.iterate(2)
    _check_orders(recorder, BUCKETS if annihilation else HASH)
    b.close()


def test_negative_record_count_is_refused(recorder):
    """hande_estimators with max < 0 must not hand back records already fetched."""
    g = hande.Hande(*_run(0), stream=1, torch_memory=False)
    g.iterate(5)
    n = C.c_int(7)
    assert recorder.hande_estimators(g._h, None, -2, C.byref(n)) == -1
    assert len(g.estimators()["iter"]) == 5
    assert recorder.hande_estimators(g._h, None, -2, C.byref(n)) == -1
    assert len(g.estimators()["iter"]) == 0
    g.close()


@pytest.mark.parametrize("width,m,n,k,ldd,shift", SHAPES)
def test_gemm_tile_width_and_store_path(recorder, width, m, n, k, ldd, shift):
    recorder.fake_reset()
    pad = (k + 7) // 8 * 8
    assert recorder.hande_gemm_bf16(4096, pad, 8192, pad, 4 * shift + 16384, ldd, m, n, k, 512, 1) == 0
    name = recorder.fake_name(recorder.fake_count() - 1).decode()
    tma = shift % 4 == 0 and ldd % 4 == 0 and n % 4 == 0   # the kernel with the staged TMA store (2), or without (0)
    assert f"k_gemm_bf16_tn_pILi{width}ELi{2 if tma else 0}E" in name


def test_creating_a_context_page_locks_nothing(recorder):
    """The host block of the read-backs becomes page-locked with use, once."""
    recorder.fake_reset()
    g = hande.Hande(*_run(0), stream=1, torch_memory=False)
    assert recorder.fake_host_allocs() == 0
    assert recorder.fake_device_allocs() < 60
    for _ in range(40):
        g.iterate(1)
        assert len(g.estimators()["iter"]) == 1
    assert recorder.fake_host_allocs() == 1
    g.close()
    assert recorder.fake_host_allocs() == 0
