"""Deterministic spaces whose size is at the edges of the CSR build's steps of 32
columns (and larger than the list), for every system and key width, against the
oracle bit for bit: the projection's sums are exact, so the tolerance is zero."""
from __future__ import annotations

import pytest

import oracle
from paper_1811_11679_gb300 import hande, inputs
from test_gpu_parity import _same_lists, _same_records

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("size", [1, 2, 31, 32, 33, 64, 65, 500, 5000])
@pytest.mark.parametrize("make,tau", [
    (lambda: inputs.hubbard_lattice_system([[3, 3], [3, -3]], 9, 9, 1.0, 1.3), 0.002),
    (lambda: inputs.molecule_system(), 0.01),
    (lambda: inputs.ueg_system(14, 19, 1.0), 0.002),     # one, two, three and eight words
    (lambda: inputs.ueg_system(14, 38, 1.0), 0.002),
    (lambda: inputs.ueg_system(14, 66, 1.0), 0.002),
    (lambda: inputs.ueg_system(10, 97, 1.0), 0.001)])
def test_core_sizes(make, tau, size):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)
    sysd = make()
    q = inputs.qmc_params(tau=tau, target_population=1e6, initiator=1, real_amplitudes=1, spawn_cutoff=0.1,
                          init_pop=2000, seed=4, semi_stoch_size=size, semi_stoch_start=6, state_capacity=60_000,
                          spawn_capacity=120_000)
    g, c = hande.Hande(sysd, q), oracle.Oracle(sysd, q)
    for step in (6, 1, 4):
        g.iterate(step)
        c.iterate(step)
        n = _same_lists(g, c, g.iterations)
    assert n > 33
    _same_records(g, c)
    assert 0 < g.diagnostics()["ncore"] <= size
    g.close()
