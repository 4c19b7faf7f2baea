"""The default annihilation (flat hash table, merge_hash.cuh) at the sizes where
it can go wrong, against the oracle bit for bit: list lengths at the edges of
its groups of 64 and tiles of 1024 entries and of the four-key search nodes, and
a one-determinant list whose surviving new determinants exceed what one group
ranks by counting (sorted runs take over).  Everything compared is an integer or
an identically ordered FP64 sum, so the tolerance is zero."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from paper_1811_11679_gb300 import hande, inputs
from test_gpu_parity import _same_lists, _same_records

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)


@pytest.mark.parametrize("norb", [19, 38, 66])     # 64-, 128- and 512-bit keys
@pytest.mark.parametrize("ndet", [2, 63, 64, 65, 1023, 1024, 1025, 16385])
def test_list_lengths_at_group_and_tile_edges(norb, ndet):
    sysd = inputs.ueg_system(14, norb, 1.0)
    q = inputs.qmc_params(tau=0.002, target_population=1e6, initiator=1, real_amplitudes=1, spawn_cutoff=0.1,
                          seed=3, state_capacity=60_001, spawn_capacity=120_000)
    keys, pops = inputs.synthetic_walkers(sysd, ndet, 3.0 * ndet + 50.0)
    g, c = hande.Hande(sysd, q), oracle.Oracle(sysd, q)
    g.set_walkers(keys, pops)
    c.set_walkers(keys, pops)
    for it in range(3):
        g.iterate(1)
        c.iterate(1)
        _same_lists(g, c, it + 1)
    _same_records(g, c)
    g.close()


@pytest.mark.parametrize("make,tau,init_pop", [
    (lambda: inputs.molecule_system(), 0.01, 1e6),             # 1309 survivors after the first iteration
    (lambda: inputs.ueg_system(14, 64, 0.5), 0.002, 2e5),      # 2001
    (lambda: inputs.ueg_system(30, 66, 1.0), 0.002, 2e5)])     # 5755
def test_group_larger_than_the_counting_limit(make, tau, init_pop):
    """tile_capacity = 64: more than 16 x 64 survivors in one group of entries
    (here all behind or before the single listed determinant) are ranked through
    sorted runs of 512."""
    sysd = make()
    q = inputs.qmc_params(tau=tau, target_population=1e7, initiator=1, real_amplitudes=1, spawn_cutoff=0.1,
                          init_pop=init_pop, seed=7, tile_capacity=64, state_capacity=400_000, spawn_capacity=800_000)
    g, c = hande.Hande(sysd, q), oracle.Oracle(sysd, q)
    largest = 0
    for it in range(2):
        g.iterate(1)
        c.iterate(1)
        largest = max(largest, g.diagnostics()["max_bucket_spawns"])
        _same_lists(g, c, it + 1)
    _same_records(g, c)
    assert largest > 16 * 64
    g.close()


@pytest.mark.parametrize("norb", [65, 96, 97])   # 130, 192 (three device words) and 194 bits (eight)
def test_wide_keys_at_the_three_word_limit(norb):
    sysd = inputs.ueg_system(10, norb, 1.0)
    assert sysd["key_words"] == 8
    q = inputs.qmc_params(tau=0.001, target_population=1e6, initiator=1, real_amplitudes=1, spawn_cutoff=0.1,
                          init_pop=2000, seed=5, state_capacity=50_001, spawn_capacity=100_000)
    g, c = hande.Hande(sysd, q), oracle.Oracle(sysd, q)
    for it in range(12):
        g.iterate(1)
        c.iterate(1)
        _same_lists(g, c, it + 1)
    _same_records(g, c)
    k, p, h, _ = g.walkers()
    g2 = hande.Hande(sysd, q)
    g2.set_walkers(k, p)
    k2, p2, h2, _ = g2.walkers()
    assert np.array_equal(k, k2) and np.array_equal(p, p2) and np.array_equal(h, h2)
    bad = k.copy()
    bad[-1, 7] |= np.uint64(1) << np.uint64(63)    # beyond the spin orbitals
    with pytest.raises(hande.HandeError):
        g2.set_walkers(bad, p)
    g.close()
    g2.close()
