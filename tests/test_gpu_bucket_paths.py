"""The bucket annihilation (annihilation = 1: block tiles, 2: one warp per bucket)
against the oracle, chosen explicitly: bucket counts beyond one chunk of 4096 of
the one-block scans, batches (their own kernels), the deterministic space chosen
mid-run, and the autotuners, which here do change the bucket sizes.  Integers and
identically ordered FP64 sums are compared: the tolerance is zero."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from paper_1811_11679_gb300 import hande, inputs
from test_gpu_batch import _mixed_replicas
from test_gpu_large_buckets import CASES, SCAN_CHUNK
from test_gpu_parity import _same_lists, _same_records

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)


def _on_bucket_path(g):
    """nbuckets and bucket_main come from the splitter kernel alone there: the
    hash path writes 64 entries per group whatever the spawns."""
    d = g.diagnostics()
    assert d["bucket_main"] != 64
    assert _launches(g) >= 9   # the hash path has six
    return d


def _launches(g):
    """Kernels of an iteration without the deterministic space's three."""
    d = g.diagnostics()
    return d["launches_per_iteration"] - (3 if d["ncore"] > 0 else 0)


@pytest.mark.parametrize("annihilation", [1, 2])
@pytest.mark.parametrize("case", sorted(CASES))
def test_many_buckets(case, annihilation):
    spec = CASES[case]
    sysd, q = spec["system"](), inputs.qmc_params(**spec["qmc"], annihilation=annihilation)
    keys, pops = inputs.synthetic_walkers(sysd, spec["ndet"], spec["walkers"])
    g, c = hande.Hande(sysd, q), oracle.Oracle(sysd, q)
    g.set_walkers(keys, pops)
    c.set_walkers(keys, pops)
    counts = []
    for it in range(2):
        g.iterate(1)
        c.iterate(1)
        counts.append(_on_bucket_path(g)["nbuckets"])
        _same_lists(g, c, it + 1)
    if annihilation == 2 and sysd["key_words"] < 8:
        assert max(counts) > SCAN_CHUNK, counts
    _same_records(g, c)
    g.close()


@pytest.mark.parametrize("annihilation", [1, 2])
def test_mixed_batch(annihilation):
    """Every replica on the bucket path but one, which stays on the hash path."""
    runs = [(s, dict(q, annihilation=annihilation)) for s, q in _mixed_replicas()]
    wide = inputs.ueg_system(14, 66, 1.0)
    runs.append((wide, inputs.qmc_params(tau=0.002, target_population=1e6, initiator=1, real_amplitudes=1,
                                         spawn_cutoff=0.1, init_pop=3000, seed=7, annihilation=annihilation)))
    runs.append(_mixed_replicas()[3])
    b = hande.HandeBatch([s for s, _ in runs], [q for _, q in runs])
    cs = [oracle.Oracle(s, q) for s, q in runs]
    done = 0
    for step in (1, 4, 30, 25):   # molecule28's deterministic space comes at iteration 40
        b.iterate(step)
        done += step
        for r, (g, c) in enumerate(zip(b.replicas, cs)):
            c.iterate(step)
            _same_lists(g, c, f"{done} (replica {r})")
    for r, (g, c) in enumerate(zip(b.replicas, cs)):
        _same_records(g, c)
        if r < len(runs) - 1:
            assert _launches(g) >= 9
    assert b.replicas[-1].diagnostics()["bucket_main"] == 64
    assert b.replicas[5].diagnostics()["ncore"] > 0
    b.close()


@pytest.mark.parametrize("annihilation", [1, 2])
def test_large_lists_in_a_batch(annihilation):
    """128- and 512-bit replicas with hundreds of buckets each."""
    runs, lists = [], []
    for r, (norb, ndet) in enumerate([(66, 40000), (66, 20000), (38, 30000)]):
        s = inputs.ueg_system(14, norb, 1.0)
        runs.append((s, inputs.qmc_params(tau=0.002, target_population=1e7, initiator=1, real_amplitudes=1,
                                          spawn_cutoff=0.1, seed=5 + r, annihilation=annihilation,
                                          state_capacity=400_000, spawn_capacity=800_000)))
        lists.append(inputs.synthetic_walkers(s, ndet, 3.0 * ndet, seed=30 + r))
    b = hande.HandeBatch([s for s, _ in runs], [q for _, q in runs])
    cs = [oracle.Oracle(s, q) for s, q in runs]
    for g, c, (k, p) in zip(b.replicas, cs, lists):
        g.set_walkers(k, p)
        c.set_walkers(k, p)
    for it in range(2):
        b.iterate(1)
        for r, (g, c) in enumerate(zip(b.replicas, cs)):
            c.iterate(1)
            _same_lists(g, c, f"{it + 1} (replica {r})")
    for g, c in zip(b.replicas, cs):
        assert _on_bucket_path(g)["nbuckets"] > (256 if annihilation == 2 else 100)   # block tiles are larger
        _same_records(g, c)
    b.close()


@pytest.mark.parametrize("annihilation", [1, 2])
def test_autotuners_keep_the_lists(annihilation):
    s, q = inputs.workload("ueg14", target_population=20000, init_pop=2000, annihilation=annihilation)
    g, c = hande.Hande(s, q), oracle.Oracle(s, q)
    g.iterate(20)
    assert g.autotune(iterations=1)["bucket_spawns"] >= 1
    g.iterate(4)
    c.iterate(g.iterations)
    _same_lists(g, c, g.iterations)
    g.close()
    b = hande.HandeBatch([s, s], [q, dict(q, seed=9)])
    b.iterate(20)
    b.autotune(iterations=1)
    b.iterate(3)
    for r, v in enumerate(b.replicas):
        c = oracle.Oracle(s, dict(q, seed=9) if r else q)
        c.iterate(v.iterations)
        _same_lists(v, c, v.iterations)
    b.close()
