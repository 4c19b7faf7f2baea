"""Diagonal elements on both sides of the electron number up to which the
annihilation lists a new determinant's orbitals in shared memory (32), beyond
which they come from the bit string, for every key width, against the oracle
bit for bit: of the determinants that an iteration adds and of a list set from
the host.  The FP64 sums are ordered alike, so the tolerance is zero."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from paper_1811_11679_gb300 import hande, inputs
from test_gpu_parity import _same_lists, _same_records

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nel", [32, 33, 34])
@pytest.mark.parametrize("make", [lambda nel: inputs.molecule_system(24, nel // 2, nel - nel // 2),   # 64-bit keys
                                  lambda nel: inputs.ueg_system(nel, 38, 1.0),                        # 128
                                  lambda nel: inputs.ueg_system(nel, 66, 1.0),                        # three words
                                  lambda nel: inputs.ueg_system(nel, 97, 1.0)])                       # eight
def test_diagonal_elements_at_the_listing_limit(make, nel):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)
    sysd = make(nel)
    q = inputs.qmc_params(tau=2e-4, target_population=1e6, initiator=1, real_amplitudes=1, spawn_cutoff=0.05, seed=3,
                          state_capacity=60_001, spawn_capacity=120_000)
    keys, pops = inputs.synthetic_walkers(sysd, 500, 8000.0)
    g, c = hande.Hande(sysd, q), oracle.Oracle(sysd, q)
    g.set_walkers(keys, pops)
    c.set_walkers(keys, pops)
    _same_lists(g, c, 0)
    n = 0
    for it in range(3):
        g.iterate(1)
        c.iterate(1)
        n = _same_lists(g, c, it + 1)
    assert n > 500   # new determinants came
    _same_records(g, c)
    g.close()
