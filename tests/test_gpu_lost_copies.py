"""FP64 launches that the host does not wait for (a launch per step, pairs of
steps, the batch's ticks, a launch per transposed step) take their tables by copies
with bounded waits.  A wait that ran out is reported by the next call that waits for
the stream; injected on the host here, by setting the launches' error word behind
them (the wait itself runs out in test_gpu_bounded_wait.py, by a copy that nothing
starts)."""
import numpy as np
import pytest

from inputs import Workload, initial_planes

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_1010_3816_gb300 as tk
    tk.load_library()


W = Workload(name="lost", a=0.7, m=2, rs_min=-30.0, rs_max=70.0, Nr=801, Ntheta=40, dt=1 / 32, substeps=2, center=5.0,
             width=3.0, noise=1e-3, seed=8, observers=((10.0, 1.2),))


def _solver(mode):
    import paper_1010_3816_gb300 as tk
    g = tk.Solver(rstar_min=W.rs_min, rstar_max=W.rs_max, Nr=W.Nr, Ntheta=W.Ntheta, dt=W.dt, substeps=W.substeps)
    g.precompute(W.a, W.M, W.s, W.m)
    g.set_steps_per_launch(mode)
    g.set_initial(*initial_planes(W))
    return g, g.add_observer(*W.observers[0])


CALLS = {"state": lambda tk, g, k: g.state(), "waveform": lambda tk, g, k: g.waveform(k),
         "finite": lambda tk, g, k: tk.tk_check_finite(g.h), "synchronize": lambda tk, g, k: tk.tk_synchronize(g.h)}


@pytest.mark.parametrize("n", [3, 200])          # launched one by one; replayed from a graph
@pytest.mark.parametrize("mode", [1, 2, "batch"])
@pytest.mark.parametrize("call", sorted(CALLS))
def test_reported_once_and_the_state_is_invalid_until_set(mode, n, call):
    import paper_1010_3816_gb300 as tk
    g, k = _solver(1 if mode == "batch" else mode)
    b = tk.Batch([g]) if mode == "batch" else None
    step = b.step if b else g.step
    step(n)
    start = g.state()
    step(n)
    want = g.state()
    tk.tk_set_state(g.h, start)
    tk.tk_inject_wait_timeout(g.h)
    step(n)
    with pytest.raises(tk.TkError) as e:
        CALLS[call](tk, g, k)
    assert e.value.status == tk.TK_ERR_INTERNAL
    for again in (lambda: g.step(1), g.state):
        with pytest.raises(tk.TkError) as e:
            again()
        assert e.value.status == tk.TK_ERR_STATE
    tk.tk_set_state(g.h, start)
    step(n)
    CALLS[call](tk, g, k)
    assert np.array_equal(g.state(), want)
    if b:
        b.close()
    g.close()


def test_a_state_set_anew_is_not_blamed():
    """The word belongs to the state that the failed launches stepped."""
    import paper_1010_3816_gb300 as tk
    g, _ = _solver(1)
    s0 = g.state()
    g.step(3)
    want = g.state()
    tk.tk_set_state(g.h, s0)
    tk.tk_inject_wait_timeout(g.h)
    g.step(3)
    tk.tk_set_state(g.h, s0)
    g.step(3)
    assert np.array_equal(g.state(), want)
    g.close()


@pytest.mark.parametrize("device", [False, True])
def test_adjoint_reports_and_leaves_the_state(device):
    import torch

    import paper_1010_3816_gb300 as tk
    g, _ = _solver(1)
    g.step(4)
    s = g.state()
    dL = np.random.default_rng(1).standard_normal(s.shape)
    want = np.empty_like(s)
    g.adjoint(want, dL_dfinal=dL, independent_pi=True)
    tk.tk_inject_wait_timeout(g.h)
    with pytest.raises(tk.TkError) as e:
        if device:
            grad = torch.empty(s.shape, dtype=torch.float64, device="cuda")
            g.adjoint(grad, dL_dfinal=torch.from_numpy(dL).cuda(), independent_pi=True)
            tk.tk_synchronize(g.h)
        else:
            g.adjoint(np.empty_like(s), dL_dfinal=dL, independent_pi=True)
    assert e.value.status == tk.TK_ERR_INTERNAL
    assert np.array_equal(g.state(), s)
    got = np.empty_like(s)
    g.adjoint(got, dL_dfinal=dL, independent_pi=True)
    assert np.array_equal(got, want)
    g.close()
