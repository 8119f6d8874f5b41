"""Device memory around the adjoint: what a recorded run holds, what the sweep
holds, and that it is given back."""
import numpy as np
import pytest

from paper_2204_03756_gb300 import mtpt

pytestmark = pytest.mark.gpu

MB = 1 << 20


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2204_03756_gb300 import build
    build.build()
    mtpt.load()


def _free():
    import torch
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def _recorded(n=20000, steps=40, every=40):
    rng = np.random.default_rng(1)
    L = float(np.sqrt(n))
    p = mtpt.Params(dim=2, D=0.5, kappa=0.5, dt=0.1, lo=(0.0, 0.0), hi=(L, L), seed=4)
    h = mtpt.mtpt_create(p)
    mtpt.mtpt_set_particles(h, 2, rng.uniform(0.0, L, size=(2, n)), rng.uniform(0.0, 1.0, n))
    before = _free()
    mtpt.mtpt_adjoint_forward(h, steps, every)
    return h, before


def test_the_tape_is_held_for_the_sweep_alone():
    """A recording holds its snapshots, (steps / every + every + 1) of
    16 dim + 12 bytes per particle, tangents and per-particle scratch; the tape
    (some 250 bytes per particle and step) is the sweep's and goes with it."""
    import torch
    n, steps = 20000, 40
    g = torch.ones(n, dtype=torch.float64, device="cuda")
    g0 = torch.empty_like(g)
    h, before = _recorded(n, steps, steps)
    try:
        recorded = _free()
        snapshots = (1 + steps + 1) * 44 * n
        assert before - recorded < snapshots + 60 * MB
        mtpt.mtpt_adjoint_backward(h, g, g0)
        assert _free() >= recorded - 4 * MB
        mtpt.mtpt_adjoint_backward(h, g, g0)
        assert _free() >= recorded - 4 * MB
    finally:
        mtpt.mtpt_destroy(h)


def _sweep(p, pos, mass, g, steps, every, without_tape, retune=None):
    import torch
    h = mtpt.mtpt_create(p)
    try:
        mtpt.mtpt_set_particles(h, p.dim, pos, mass)
        mtpt.mtpt_adjoint_forward(h, steps, every)
        if retune:
            mtpt.mtpt_set_tuning(h, retune, 128)
        gt = torch.from_numpy(g).cuda()
        g0 = torch.empty_like(gt)
        mtpt.mtpt_debug_fail_alloc(-1 if without_tape else 0)
        dD = mtpt.mtpt_adjoint_backward(h, gt, g0)
        assert mtpt.mtpt_debug_fail_alloc(0) == 0     # (the injection met the tape)
        return dD, g0.cpu().numpy(), mtpt.mtpt_get_info(h)
    finally:
        mtpt.mtpt_debug_fail_alloc(0)
        mtpt.mtpt_destroy(h)


@pytest.mark.parametrize("form", [mtpt.MTPT_FP64, mtpt.MTPT_FP32W])
@pytest.mark.parametrize("clump", [0, 150])
@pytest.mark.parametrize("dim,n,L", [(1, 700, 300.0), (2, 5001, 70.0), (3, 1500, 12.0)])
def test_gradients_do_not_depend_on_free_memory(form, clump, dim, n, L):
    """With the tape, without the memory for it, and with a clump that the tape
    cannot hold: the same bits."""
    rng = np.random.default_rng(n + clump)
    pos = rng.uniform(0.0, L, size=(dim, n))
    pos[:, :clump] = L / 2 + rng.uniform(-0.2, 0.2, size=(dim, clump))
    mass, g = rng.uniform(0.0, 1.0, n), rng.uniform(-1.0, 1.0, n)
    p = mtpt.Params(dim=dim, D=0.5, kappa=0.5, dt=0.1, lo=(0.0,) * dim, hi=(L,) * dim, seed=3,
                    precision=form)
    for steps, every in ((5, 5), (7, 3)):
        taped, plain = (_sweep(p, pos, mass, g, steps, every, w) for w in (False, True))
        assert taped[0] == plain[0]
        assert np.array_equal(taped[1], plain[1])
        # a segment that the tape cannot hold is taken again, its pairs counted once
        assert taped[2]["pair_count"] == plain[2]["pair_count"]


def test_a_run_that_is_not_differentiated_holds_no_memory():
    """Under no_grad, and with a graph that is dropped before its backward."""
    import gc

    import torch
    from paper_2204_03756_gb300 import autograd
    n, L = 20000, 141.0
    rng = np.random.default_rng(2)
    p = mtpt.Params(dim=2, D=0.5, kappa=0.5, dt=0.1, lo=(0.0, 0.0), hi=(L, L), seed=4)
    pos = torch.from_numpy(rng.uniform(0.0, L, size=(2, n))).cuda()
    mass = torch.from_numpy(rng.uniform(0.0, 1.0, n)).cuda().requires_grad_()
    D = torch.tensor(0.5, requires_grad=True)

    def run(grad):
        with torch.set_grad_enabled(grad):
            m, _ = autograd.mtpt_run(mass, D, p, pos, 30, 30)
        del m
        gc.collect()

    run(False)
    level = _free()
    for grad in (False, True) * 3:          # 32 snapshots of 0.9 MB each
        run(grad)
        assert _free() >= level - 4 * MB
    # and a differentiated one
    m, _ = autograd.mtpt_run(mass, D, p, pos, 30, 30)
    m.sum().backward()
    del m
    gc.collect()
    assert _free() >= level - 4 * MB


@pytest.mark.parametrize("retune", [0.5, 2.0])
def test_a_grid_retuned_before_the_sweep_keeps_its_tape(retune):
    rng = np.random.default_rng(9)
    n, L = 1800, 42.0
    pos, mass, g = rng.uniform(0.0, L, size=(2, n)), rng.uniform(0.0, 1.0, n), rng.uniform(-1.0, 1.0, n)
    p = mtpt.Params(dim=2, D=0.5, kappa=0.5, dt=0.1, lo=(0.0, 0.0), hi=(L, L), seed=4)
    taped, plain = (_sweep(p, pos, mass, g, 8, 8, w, retune) for w in (False, True))
    assert taped[0] == plain[0] and np.array_equal(taped[1], plain[1])


@pytest.mark.parametrize("steps,met", [(1, False), (4, False), (5, True)])
def test_short_sweeps_take_no_tape(steps, met):
    """Below five steps the tape's allocation costs more than it spares."""
    import torch
    h, _ = _recorded(2000, steps, 20)
    try:
        g = torch.ones(2000, dtype=torch.float64, device="cuda")
        mtpt.mtpt_debug_fail_alloc(-1)
        mtpt.mtpt_adjoint_backward(h, g, torch.empty_like(g))
        assert (mtpt.mtpt_debug_fail_alloc(0) == 0) == met
    finally:
        mtpt.mtpt_debug_fail_alloc(0)
        mtpt.mtpt_destroy(h)
