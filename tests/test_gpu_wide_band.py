"""Boxes in which the band of the pair test is wider than the cutoff: cells some
1e5 cutoffs wide (a cloud in a large domain) and coordinates 1e13 cutoffs from the
origin, where binary32 offsets decide no pair and every candidate gets the exact
test.  Pair counts equal the oracle's in every form; the binary64 form's masses
too; the precision form's row sums as far as its offsets allow."""
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


def _case(dim, where, form, n):
    """(params, positions): `just` a half-width just above psi^2, `wide` many
    times it, `far` a box far from the origin."""
    rng = np.random.default_rng(dim)
    psi = 3.0 * np.sqrt(4.0 * 5e-10)
    # the cells are capped at about 4 n + 64, so this is their width in cutoffs
    side = {"just": {1: 1.6e4, 2: 1020.0, 3: 307.0}, "wide": {1: 1e8, 2: 1e6, 3: 1e5}}
    if where == "far":
        lo, side, D = 1e13, 100.0, 1.0 / 36.0
        pos = lo + rng.uniform(0.0, side if dim < 3 else 12.0, size=(dim, n))
    else:
        lo, side, D = 0.0, side[where][dim], 5e-10
        clump = psi * {1: 200.0, 2: 20.0, 3: 8.0}[dim]
        pos = side * 0.37 + rng.uniform(0.0, clump, size=(dim, n))
        pos[:, :50] = rng.uniform(0.0, side, size=(dim, 50))
    p = mtpt.Params(dim=dim, D=D, kappa=0.0, dt=1.0, lo=(lo,) * dim, hi=(lo + side,) * dim, seed=3,
                    precision=form)
    return p, pos


def _brute(p, pos):
    d = O.derived(oracle_params(p))
    return O.pairs(pos, d["psi2"], "brute"), d


@pytest.mark.parametrize("where", ["just", "wide", "far"])
@pytest.mark.parametrize("dim", [1, 2, 3])
@pytest.mark.parametrize("form", FORMS)
def test_pairs_are_exact(form, dim, where):
    n = 2050
    p, pos = _case(dim, where, form, n)
    mass = np.random.default_rng(4).uniform(0.0, 1.0, n)
    (bi, bj), d = _brute(p, pos)
    with mtpt.Simulation(p, pos, mass) as sim:
        sim.step(2)                               # kappa = 0: the particles stay
        info, got, rows = sim.info(), sim.masses(), sim.row_sums() / d["kernel_norm"]
        gi, gj = sim.pairs()
    assert info["pair_count"] == 2 * len(bi)
    assert np.array_equal(gi, bi) and np.array_equal(gj, bj)
    if form == mtpt.MTPT_FP64:
        _, want, _ = O.run(oracle_params(p), pos, mass, 2)
        assert rel_err(got, want) <= TOL[form]
        return
    # every flux is antisymmetric: the total stays, to binary32 sums
    assert got.sum() == pytest.approx(mass.sum(), rel=1e-6)
    if where != "just":
        return
    # an offset from the cell's corner is off by its last rounding, at most u w
    # (u = 2^-24; the clump lies inside one cell), so with e = 2 u w per axis d2 is
    # within delta = sum_a (2 |dx_a| e + e^2) and K within a factor exp(a delta)
    a, w, u = 1.0 / (2.0 * d["h2"]), np.asarray(info["cell_width"][:dim]), 2.0 ** -24
    e = 2.0 * u * w
    dx = np.abs(pos[:, bi] - pos[:, bj])
    d2 = (dx ** 2).sum(axis=0)
    K = np.exp(-a * d2)
    delta = (2.0 * dx * e[:, None] + e[:, None] ** 2).sum(axis=0)
    want, slack = np.ones(n), np.full(n, 1e-5)
    np.add.at(want, bi, K)
    np.add.at(slack, bi, K * np.expm1(a * delta) + 1e-6)
    assert np.all(np.abs(rows - want) <= slack)
    # ... which for most particles is less than a second K from every pair beyond
    # the half-width's excess over psi^2 would add
    dc = 3.0 * u * 2.0 * p.hi[0] / d["psi"]
    eta = 2.0 * 14.0 * u * (1.0 + dc) * w.sum() / d["psi"]
    assert 1.0 < eta < 1.1
    twice = np.zeros(n)
    np.add.at(twice, bi, np.where(d2 > (eta - 1.0) * d["psi2"], K, 0.0))
    assert np.mean(twice > slack) > 0.9


def test_batch_and_no_allocation_step_share_the_search():
    """Realisations with and without such a band in one batch, and the step on
    caller's buffers."""
    import torch
    n = 2050
    p, pos = _case(2, "just", mtpt.MTPT_FP32W, n)
    q = mtpt.Params(dim=2, D=1.0, kappa=0.0, dt=0.1, lo=(0.0, 0.0), hi=(45.0, 45.0), seed=5,
                    precision=mtpt.MTPT_FP32W)
    rng = np.random.default_rng(8)
    qpos, m = rng.uniform(0.0, 45.0, size=(2, n)), rng.uniform(0.0, 1.0, n)
    alone = []
    for prm, x in ((p, pos), (q, qpos)):
        with mtpt.Simulation(prm, x, m) as sim:
            sim.step(2)
            alone.append(sim.masses())
    with mtpt.Batch([p, q], [n, n], np.concatenate([pos, qpos], axis=1), np.concatenate([m, m])) as b:
        b.step(2)
        assert np.array_equal(b.masses(), np.concatenate(alone))
    xt, mt = torch.from_numpy(pos.copy()).cuda(), torch.from_numpy(m.copy()).cuda()
    for call in range(2):
        mtpt.mtpt_step_noalloc(p, call, xt, mt)
    torch.cuda.synchronize()
    assert np.array_equal(mt.cpu().numpy(), alone[0])
