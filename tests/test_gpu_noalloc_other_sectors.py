"""hande_estimate_noalloc on keys of another electron-number sector.  The header
does not ask for the context's electron numbers, and a UEG element between
determinants that differ in two spin orbitals is zero: such keys add to the
walker number and nothing else, whichever side the two orbitals are on.
Integers are compared, so the tolerance is zero."""
from __future__ import annotations

import numpy as np
import pytest

from paper_1811_11679_gb300 import hande, inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("norb", [19, 38, 66])   # 1, 2 and 8 key words
def test_keys_two_orbitals_from_the_reference(norb):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)
    sysd = inputs.ueg_system(14, norb, 1.0)
    g = hande.Hande(sysd, inputs.qmc_params(tau=0.002, target_population=1e4, initiator=1, real_amplitudes=1,
                                            spawn_cutoff=0.1, init_pop=100, seed=7, state_capacity=5000,
                                            spawn_capacity=10000))
    keys, pops = inputs.synthetic_walkers(sysd, 2000, 6000.0)
    _, d0 = g.reference()
    bit = lambda p: int(d0[p >> 6]) >> (p & 63) & 1
    occ = [p for p in range(2 * norb) if bit(p)]
    emp = [p for p in range(2 * norb) if not bit(p)]

    def flipped(*orbitals):
        k = d0.copy()
        for p in orbitals:
            k[p >> 6] ^= np.uint64(1) << np.uint64(p & 63)
        return k

    other = np.array([flipped(emp[0], emp[1]), flipped(emp[0], emp[-1]),       # two electrons more
                      flipped(occ[0], occ[1]), flipped(occ[0], occ[-1]),       # two fewer
                      flipped(occ[0], emp[0]), flipped(occ[-1], emp[-1])])     # one moved
    extra = np.arange(1, len(other) + 1, dtype=np.int64) << 32

    def sums(k, p):
        dk = torch.from_numpy(np.ascontiguousarray(k).view(np.int64)).cuda()
        dp = torch.from_numpy(np.ascontiguousarray(p)).cuda()
        out = torch.full((4,), -1, dtype=torch.int64, device="cuda")
        torch.cuda.synchronize()
        g.estimate_noalloc(dk.data_ptr(), dp.data_ptr(), len(p), out.data_ptr())
        g.synchronize()
        return out.cpu().numpy()

    want = sums(keys, pops)
    assert want[2] != 0 or want[3] != 0
    got = sums(np.concatenate([keys, other]), np.concatenate([pops, extra]))
    want[0] += extra.sum()
    assert np.array_equal(got, want)
    g.close()
