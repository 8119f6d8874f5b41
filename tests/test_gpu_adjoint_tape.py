"""The adjoint sweep on and off its tape: runs whose neighbours fit the tape's
mask words and values, runs with a clump that does not (the sweep then takes
that segment step by step), one tile of a warp and ragged ends, 1-d to 3-d, and
a grid retuned between recording and sweep; against the oracle's reverse sweep,
and the two ways against each other."""
import numpy as np
import pytest

import oracle as O
from paper_2204_03756_gb300 import mtpt

from gpu_helpers import oracle_params, rel_err

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2204_03756_gb300 import build
    build.build()
    mtpt.load()


def _reverse(p, pos, n, steps, g):
    op, ids, xs, x = oracle_params(p), np.arange(n, dtype=np.uint32), [], pos
    for t in range(steps):
        x = O.random_walk(op, x, ids, t)
        xs.append(x)
    for t in reversed(range(steps)):
        g = O.mass_transfer(op, xs[t], g)[0]
    return g


def _sweep(p, pos, mass, steps, every, g, retune=None):
    import torch
    h = mtpt.mtpt_create(p)
    try:
        mtpt.mtpt_set_particles(h, p.dim, pos, mass)
        mtpt.mtpt_adjoint_forward(h, steps, every)
        if retune:
            mtpt.mtpt_set_tuning(h, retune, 128)
        gt = torch.from_numpy(g).cuda()
        g0 = torch.empty_like(gt)
        dD = mtpt.mtpt_adjoint_backward(h, gt, g0)
        return g0.cpu().numpy(), dD
    finally:
        mtpt.mtpt_destroy(h)


@pytest.mark.parametrize("form", [mtpt.MTPT_FP64, mtpt.MTPT_FP32W])
@pytest.mark.parametrize("dim,n,L,clump", [(1, 33, 30.0, 0), (1, 700, 300.0, 0), (1, 700, 300.0, 150),
                                           (2, 255, 16.0, 0), (2, 2049, 45.0, 0), (2, 2049, 45.0, 150),
                                           (3, 1500, 12.0, 0), (3, 1500, 12.0, 150)])
def test_sweep_on_and_off_the_tape(form, dim, n, L, clump):
    rng = np.random.default_rng(n + clump)
    pos = rng.uniform(0.0, L, size=(dim, n))
    pos[:, :clump] = L / 2 + rng.uniform(-0.2, 0.2, size=(dim, clump))
    mass, g = rng.uniform(0.0, 1.0, n), rng.uniform(-1.0, 1.0, n)
    p = mtpt.Params(dim=dim, D=0.5, kappa=0.5, dt=0.1, lo=(0.0,) * dim, hi=(L,) * dim, seed=3,
                    precision=form)
    steps = 5
    want = _reverse(p, pos, n, steps, g)
    got = [_sweep(p, pos, mass, steps, every, g) for every in (5, 2, 1)]
    for g0, dD in got:
        assert rel_err(g0, want) <= 1e-12
        # the same sums in another grouping; the forward masses are the same
        assert abs(dD - got[0][1]) <= 1e-10 * max(abs(dD), 1e-3)


def test_grid_retuned_between_recording_and_sweep():
    rng = np.random.default_rng(9)
    n, L = 1800, 42.0
    pos, mass, g = rng.uniform(0.0, L, size=(2, n)), rng.uniform(0.0, 1.0, n), rng.uniform(-1.0, 1.0, n)
    p = mtpt.Params(dim=2, D=0.5, kappa=0.5, dt=0.1, lo=(0.0, 0.0), hi=(L, L), seed=4)
    want = _reverse(p, pos, n, 4, g)
    for retune in (None, 0.5, 2.0):
        assert rel_err(_sweep(p, pos, mass, 4, 4, g, retune)[0], want) <= 1e-12
