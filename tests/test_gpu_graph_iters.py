"""hande_iterate(n) launches several iterations per CUDA graph where no host work
is due between them: any split of a run into calls gives the same lists and
records, also across the iteration that chooses the deterministic space."""
from __future__ import annotations

import numpy as np
import pytest

from paper_1811_11679_gb300 import hande, inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("start", [0, 6, 8, 13])
def test_any_split_into_calls_gives_the_same_run(start):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    size = 50 if start else 0
    s, q = inputs.workload("molecule28", target_population=3000, init_pop=500, semi_stoch_size=size,
                           semi_stoch_start=start)
    runs = []
    for calls in ([1] * 23, [23], [3, 4, 5, 7, 4], [4, 1, 4, 1, 8, 5]):
        h = hande.Hande(s, q)
        for n in calls:
            h.iterate(n)
        assert h.iterations == 23
        runs.append((h.walkers(), h.estimators()))
        h.close()
    for (w, r) in runs[1:]:
        for a, b in zip(w, runs[0][0]):
            assert np.array_equal(np.asarray(a).view(np.uint8), np.asarray(b).view(np.uint8))
        for k in r:
            assert np.array_equal(r[k].view(np.uint8), runs[0][1][k].view(np.uint8)), k
