"""FP64 solvers where the device's memory does not reach for the step's or the
adjoint's split tables: they run on the unsplit ones, as every grid that fits without
the split tables does, and give the same results but for roundings.

Tolerance: test_gpu_split.py's, 16 roundings of 2^-53 on either side per step and a
growth of ten.
"""
import numpy as np
import pytest

from inputs import Workload, initial_planes

pytestmark = pytest.mark.gpu

N = 6
TOL = 10 * 2 * 16 * N * 2.0 ** -53
MB = 1 << 20
W = Workload(name="mem", a=0.9, m=2, rs_min=-50.0, rs_max=750.0, Nr=25601, Ntheta=64, dt=1 / 64, center=20.0, width=4.0,
             noise=1e-3, seed=11)
POINT = W.Nr * 64
STATE, PLAIN, SPLIT, ADJ = POINT * 32, POINT * (168 + 8), POINT // 32 * 5776, POINT // 32 * 6544


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_1010_3816_gb300 as tk
    tk.load_library()


def _solver():
    import paper_1010_3816_gb300 as tk
    g = tk.Solver(rstar_min=W.rs_min, rstar_max=W.rs_max, Nr=W.Nr, Ntheta=W.Ntheta, dt=W.dt)
    g.precompute(W.a, W.M, W.s, W.m)
    return g


def _run(g, planes, dL, state, grad, mode):
    g.set_steps_per_launch(mode)
    g.set_initial(*planes)
    g.step(N - 1)
    if dL is not None:
        g.adjoint(grad, dL_dfinal=dL, independent_pi=True)
    g.step(1)
    g.state(out=state)
    return state


# what is left: the solver, the copy of its initial state that it keeps, what the
# allocations round up to, and (bytes, whether the adjoint runs too)
BASE = 3 * STATE + PLAIN + 16 * MB
LEFT = {"no step tables": (BASE + SPLIT // 2, False),
        "no adjoint tables": (BASE + SPLIT + 2 * STATE + ADJ // 2, True),
        "step tables given up for an adjoint state": (BASE + SPLIT + STATE + STATE // 2, True)}


@pytest.mark.parametrize("mode", [0, 1, 2])
@pytest.mark.parametrize("left", sorted(LEFT))
def test_grids_that_fit_without_the_split_tables(left, mode):
    import torch

    import paper_1010_3816_gb300 as tk
    bytes_left, adjoint = LEFT[left]
    dev = torch.device("cuda")
    planes = [torch.from_numpy(x).to(dev) for x in initial_planes(W)]
    dL = torch.from_numpy(np.random.default_rng(1).standard_normal((4, W.Ntheta, W.Nr))).to(dev) if adjoint else None
    state, grad = (torch.empty((4, W.Ntheta, W.Nr), dtype=torch.float64, device=dev) for _ in range(2))
    g = _solver()
    want = _run(g, planes, dL, state, grad, mode).cpu().numpy()
    want_grad = grad.cpu().numpy()
    g.close()
    torch.cuda.synchronize()
    hold = torch.empty(torch.cuda.mem_get_info()[0] - bytes_left, dtype=torch.uint8, device=dev)
    try:
        g = _solver()
        if not adjoint:
            assert torch.cuda.mem_get_info()[0] < SPLIT + STATE      # so they are not there
        got = _run(g, planes, dL, state, grad, mode).cpu().numpy()
        got_grad = grad.cpu().numpy()
        tk.tk_synchronize(g.h)
        g.close()
    finally:
        del hold
        torch.cuda.empty_cache()
    for c in range(4):
        assert np.linalg.norm(got[c] - want[c]) <= TOL * np.linalg.norm(want[c])
    if adjoint:
        assert np.linalg.norm(got_grad - want_grad) <= TOL * np.linalg.norm(want_grad)



def test_batch_with_a_member_without_the_split_tables():
    """The queue needs them of every member; the members are then stepped one after
    another, the second of these without its tables."""
    import torch

    import paper_1010_3816_gb300 as tk
    dev = torch.device("cuda")
    planes = [torch.from_numpy(x).to(dev) for x in initial_planes(W)]
    state, grad = (torch.empty((4, W.Ntheta, W.Nr), dtype=torch.float64, device=dev) for _ in range(2))
    g = _solver()
    want = _run(g, planes, None, state, grad, 0).cpu().numpy()
    g.close()
    torch.cuda.synchronize()
    hold = torch.empty(torch.cuda.mem_get_info()[0] - (2 * BASE + SPLIT + SPLIT // 4 + 2 * STATE), dtype=torch.uint8, device=dev)
    try:
        gs = [_solver(), _solver()]
        for g in gs:
            g.set_initial(*planes)
        b = tk.Batch(gs)
        b.step(2)
        seg, ms = b.tune(1)
        assert seg == 0 and ms > 0.0
        b.step(N - 2)
        got = [g.state(out=state).cpu().numpy() for g in gs]
        b.close()
        for g in gs:
            g.close()
    finally:
        del hold
        torch.cuda.empty_cache()
    assert not np.array_equal(got[0], got[1])
    for s in got:
        for c in range(4):
            assert np.linalg.norm(s[c] - want[c]) <= TOL * np.linalg.norm(want[c])
