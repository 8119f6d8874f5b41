"""What pass 1 keeps for pass 2 is memory that a run can do without: when the
device has none for it, every call still runs and gives the same results."""
import numpy as np
import pytest

from paper_2204_03756_gb300 import mtpt

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2204_03756_gb300 import build
    build.build()
    mtpt.load()
    yield
    mtpt.mtpt_debug_fail_alloc(0)


def _params(dim, form, L):
    return mtpt.Params(dim=dim, D=1.0, kappa=0.5, dt=0.1, lo=(0.0,) * dim, hi=(L,) * dim, seed=6,
                       precision=form)


def _run(p, pos, mass, nth):
    """A load, a multi-step call, a larger grid, more steps; the nth optional
    allocation fails."""
    mtpt.mtpt_debug_fail_alloc(-nth)
    with mtpt.Simulation(p, pos, mass) as sim:
        sim.step(13)
        rows = sim.row_sums()
        sim.set_tuning(0.5, 128)
        sim.step(3)
        out = sim.positions(), sim.masses(), rows, sim.info()["pair_count"]
        sim.set_tuning(1.0, 256)
        sim.step(2)
        out += (sim.masses(),)
    return out, mtpt.mtpt_debug_fail_alloc(0)


@pytest.mark.parametrize("form", [mtpt.MTPT_FP64, mtpt.MTPT_FP32W])
@pytest.mark.parametrize("dim,n,L", [(1, 3001, 3000.0), (2, 5001, 70.0), (2, 5001, 22.0), (3, 3001, 14.0)])
def test_steps(form, dim, n, L):
    rng = np.random.default_rng(dim)
    pos, mass = rng.uniform(0.0, L, size=(dim, n)), rng.uniform(0.0, 1.0, n)
    p = _params(dim, form, L)
    want, _ = _run(p, pos, mass, 0)
    for nth in range(1, 20):
        got, left = _run(p, pos, mass, nth)
        for a, b in zip(got, want):
            assert np.array_equal(a, b)
        if left:                              # one more than the run makes
            break
    assert nth > (3 if form == mtpt.MTPT_FP64 else 1)


@pytest.mark.parametrize("form", [mtpt.MTPT_FP64, mtpt.MTPT_FP32W])
def test_gradients(form):
    import torch
    n, L = 4001, 63.0
    rng = np.random.default_rng(5)
    pos, mass = rng.uniform(0.0, L, size=(2, n)), rng.uniform(0.0, 1.0, n)
    g = torch.from_numpy(rng.uniform(-1.0, 1.0, n)).cuda()
    p = _params(2, form, L)

    def run(nth):
        h = mtpt.mtpt_create(p)
        try:
            mtpt.mtpt_set_particles(h, 2, pos, mass)
            mtpt.mtpt_debug_fail_alloc(-nth)
            mtpt.mtpt_adjoint_forward(h, 7, 3)
            g0 = torch.empty_like(g)
            dD = mtpt.mtpt_adjoint_backward(h, g, g0)
            left = mtpt.mtpt_debug_fail_alloc(0)
            return (dD, g0.cpu().numpy()), left
        finally:
            mtpt.mtpt_debug_fail_alloc(0)
            mtpt.mtpt_destroy(h)

    want, _ = run(0)
    for nth in range(1, 10):
        got, left = run(nth)
        assert got[0] == want[0] and np.array_equal(got[1], want[1])
        if left:
            break
    assert nth > 3
