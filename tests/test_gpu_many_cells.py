"""A long 1-d box with more cutoffs than binary32 has whole numbers: the records hold
cell indexes in binary32, so an axis has at most 2^24 cells (wider ones then)."""
import numpy as np
import pytest

import oracle as O
from paper_2204_03756_gb300 import mtpt

from gpu_helpers import oracle_params

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2204_03756_gb300 import build
    build.build()
    mtpt.load()


@pytest.mark.parametrize("form", [mtpt.MTPT_FP64, mtpt.MTPT_FP32W])
def test_pairs_beyond_2_to_the_24_cutoffs(form):
    n = 6_000_000
    p = mtpt.Params(dim=1, D=0.1, kappa=0.0, dt=0.1, lo=(0.0,), hi=(1.3e7,), seed=1, precision=form)
    psi2 = O.derived(oracle_params(p))["psi2"]
    assert p.hi[0] / np.sqrt(psi2) > 2 ** 24
    rng = np.random.default_rng(2)
    x = np.sort(rng.uniform(0.6 * p.hi[0], p.hi[0], n))        # the far end's cells
    pairs, k = 0, 1
    while True:
        d = x[k:] - x[:-k]
        near = int(np.count_nonzero(d * d <= psi2))
        if near == 0:
            break
        pairs += 2 * near
        k += 1
    with mtpt.Simulation(p, x[None, :], np.ones(n)) as sim:
        sim.step(1)
        info = sim.info()
    assert info["pair_count"] == pairs
    assert info["cells"][0] <= 2 ** 24
