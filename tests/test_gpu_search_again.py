"""Particles whose neighbours are not kept between the two pair passes (a clump in
a large box, or no room for the words): pass 2, and in binary64 pass 1, search
again and give the same sums."""
import numpy as np
import pytest

import oracle as O
from paper_2204_03756_gb300 import mtpt

from gpu_helpers import TOL, oracle_params, rel_err

pytestmark = pytest.mark.gpu

FORMS = [mtpt.MTPT_FP64, mtpt.MTPT_FP32W]


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2204_03756_gb300 import build
    build.build()
    mtpt.load()


def _lattice(dim, k, step, at):
    g = np.stack(np.meshgrid(*[np.arange(k)] * dim, indexing="ij")).reshape(dim, -1)
    return g * step + at


# psi = 1.25 is a lattice distance, so the exact test decides many pairs; the large
# box makes the words too few
@pytest.mark.parametrize("dim,k,step,side", [(1, 401, 2.0 ** -6, 4000.0), (2, 33, 0.25, 2000.0),
                                             (3, 13, 0.25, 300.0)])
@pytest.mark.parametrize("form", FORMS)
def test_lattice_beyond_the_words(form, dim, k, step, side):
    pos = _lattice(dim, k, step, side / 2)
    n = pos.shape[1]
    mass = np.random.default_rng(dim).uniform(0.0, 1.0, n)
    p = mtpt.Params(dim=dim, D=2.5, kappa=0.0, dt=0.1, lam=1.25, lo=(0.0,) * dim, hi=(side,) * dim,
                    seed=7, precision=form)
    assert O.derived(oracle_params(p))["psi2"] == pytest.approx(1.5625)
    with mtpt.Simulation(p, pos, mass) as sim:
        sim.step(3)
        got, info = sim.masses(), sim.info()
    _, want, npairs = O.run(oracle_params(p), pos, mass, 3, method="brute")
    assert info["pair_count"] == npairs
    assert npairs > 40 * n
    assert rel_err(got, want) <= TOL[form]


@pytest.mark.parametrize("dim", [1, 2, 3])
@pytest.mark.parametrize("form", FORMS)
def test_reaction_with_a_clump(form, dim):
    """Both species through the search."""
    rng = np.random.default_rng(dim)
    n, L = 1501, {1: 900.0, 2: 60.0, 3: 20.0}[dim]
    pos = rng.uniform(0.0, L, size=(dim, n))
    pos[:, :300] = L / 2 + rng.uniform(-0.3, 0.3, size=(dim, 300))
    a, b = rng.uniform(0.0, 1.0, n), rng.uniform(0.0, 1.0, n)
    p = mtpt.Params(dim=dim, D=1.0, kappa=0.5, dt=0.1, lo=(0.0,) * dim, hi=(L,) * dim, seed=3,
                    precision=form)
    with mtpt.Simulation(p, pos, a) as sim:
        sim.set_reaction(0.7, b)
        sim.step(3)
        got = sim.masses(), sim.masses_b(), sim.info()["pair_count"]
    _, wa, wb, npairs = O.run_reactive(oracle_params(p), pos, a, b, 3, 0.7)
    assert got[2] == npairs
    assert rel_err(got[0], wa) <= TOL[form] and rel_err(got[1], wb) <= TOL[form]


@pytest.mark.parametrize("form", FORMS)
@pytest.mark.parametrize("dim,n,rho", [(3, 65535, 1.0), (3, 65535, 6.0), (2, 65535, 20.0)])
def test_no_allocation_step_without_words_equals_the_handle(form, dim, n, rho):
    """At the largest sizes the scratch has no room for the words: the same bits."""
    import torch
    rng = np.random.default_rng(n + dim)
    L = (n / rho) ** (1.0 / dim)
    pos, mass = rng.uniform(0.0, L, size=(dim, n)), rng.uniform(0.0, 1.0, n)
    p = mtpt.Params(dim=dim, D=1.0, kappa=0.5, dt=0.1, lo=(0.0,) * dim, hi=(L,) * dim, seed=3,
                    precision=form)
    x, m = torch.from_numpy(pos.copy()).cuda(), torch.from_numpy(mass.copy()).cuda()
    mtpt.mtpt_step_noalloc(p, 0, x, m)
    torch.cuda.synchronize()
    with mtpt.Simulation(p, pos, mass) as sim:
        sim.step(1)
        assert np.array_equal(x.cpu().numpy(), sim.positions())
        assert np.array_equal(m.cpu().numpy(), sim.masses())
