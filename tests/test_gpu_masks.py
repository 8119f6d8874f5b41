"""Accept masks of the precision form in 1-d and 2-d: words of 32 candidates a
neighbour row, compact or padded, against the oracle at the sizes where a word,
a row or the capacity ends (windows of about 32, 64 and 300 candidates, a clump
beyond the capacity, half-width cells, pairs exactly on the cutoff)."""
import numpy as np
import pytest

import oracle as O
from paper_2204_03756_gb300 import mtpt

from gpu_helpers import TOL, oracle_params, rel_err

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2204_03756_gb300 import build
    build.build()
    mtpt.load()


def _check(p, pos, mass, steps, cell_scale=1.0):
    with mtpt.Simulation(p, pos, mass) as sim:
        sim.set_tuning(cell_scale, 256)
        sim.step(steps)
        x, m, info = sim.positions(), sim.masses(), sim.info()
    xr, mr, npairs = O.run(oracle_params(p), pos, mass, steps)
    assert np.array_equal(x, xr)
    assert info["pair_count"] == npairs
    assert rel_err(m, mr) <= TOL[mtpt.MTPT_FP32W]


# particles per cutoff length: row windows of 2 x that many candidates in 1-d
# and about 2 x that many squared in 2-d
@pytest.mark.parametrize("dim,per_psi", [(1, 1.0), (1, 15.5), (1, 33.0), (1, 150.0), (2, 1.0),
                                         (2, 2.5), (2, 4.0), (2, 7.0)])
@pytest.mark.parametrize("cell_scale", [0.5, 1.0])
def test_windows_of_one_and_more_words(dim, per_psi, cell_scale):
    rng = np.random.default_rng(int(10 * per_psi) + dim)
    n = 3001
    psi = np.sqrt(36.0 * 0.5 * 0.1)
    L = psi * (n / per_psi ** dim) ** (1.0 / dim)
    pos = rng.uniform(0.0, L, size=(dim, n))
    mass = rng.uniform(0.0, 1.0, n)
    p = mtpt.Params(dim=dim, D=1.0, kappa=0.5, dt=0.1, lo=(0.0,) * dim, hi=(L,) * dim, seed=5,
                    precision=mtpt.MTPT_FP32W)
    _check(p, pos, mass, 3, cell_scale)


@pytest.mark.parametrize("dim", [1, 2])
def test_a_clump_beyond_the_words_searches(dim):
    rng = np.random.default_rng(dim)
    n, L = 2500, 300.0
    pos = rng.uniform(0.0, L, size=(dim, n))
    pos[:, :900] = L / 2 + rng.uniform(-0.4, 0.4, size=(dim, 900))
    p = mtpt.Params(dim=dim, D=1.0, kappa=0.5, dt=0.1, lo=(0.0,) * dim, hi=(L,) * dim, seed=6,
                    precision=mtpt.MTPT_FP32W)
    _check(p, pos, rng.uniform(0.0, 1.0, n), 2)


@pytest.mark.parametrize("kappa", [0.0, 0.5])
def test_pairs_on_the_cutoff_get_their_mask_bits(kappa):
    """A lattice with many pairs exactly psi apart (the exact test inside the
    band decides them, after the row's words are written)."""
    k = 40
    g = np.stack(np.meshgrid(np.arange(k), np.arange(k), indexing="ij")).reshape(2, -1) * 0.25 + 5.0
    p = mtpt.Params(dim=2, D=2.5 / (1.0 - kappa), kappa=kappa, dt=0.1, lam=1.25, lo=(0.0, 0.0),
                    hi=(20.0, 20.0), seed=7, precision=mtpt.MTPT_FP32W)
    assert O.derived(oracle_params(p))["psi2"] == pytest.approx(1.5625)
    _check(p, g, np.random.default_rng(8).uniform(0.0, 1.0, k * k), 1)
