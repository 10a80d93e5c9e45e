"""Columns whose coefficients are too large for the integer coupling (class sums
of 2^20 and more: "cold" tables), next to ordinary columns: they take the FP64
instructions, and their neighbours' results do not change for it.

Tolerance of one step: at most 16 roundings (2^-53 each, on terms of at most the
size of the field next to it) on either side, fields that do not grow by more
than a factor of ten.
"""
import numpy as np
import pytest

from inputs import Workload

pytestmark = pytest.mark.gpu

TOL = 10 * 2 * 16 * 2.0 ** -53
LARGE = 2.0 ** 36      # with dt = 1/64 class sums of 2^21 and more


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_1010_3816_gb300 as tk
    tk.load_library()


def _tables(Nr, Nth):
    """A workload, an oracle solver of it, and its raw coefficients as
    tk_set_coefficients takes them (the oracle's half nodes are stored one column
    to the right)."""
    import oracle
    w = Workload(name="cold", a=0.9, m=2, rs_min=-2.0, rs_max=-2.0 + (Nr - 1) / 8.0, Nr=Nr, Ntheta=Nth, dt=1 / 64)
    o = oracle.Solver(M=w.M, a=w.a, s=w.s, m=w.m, rs_min=w.rs_min, rs_max=w.rs_max, Nr=Nr, Ntheta=Nth, dt=w.dt)
    node, half = o.coeffs()
    half9 = np.zeros_like(half)
    half9[:, :, :-1] = half[:, :, 1:]
    return w, node.copy(), half9, np.stack(oracle.regular_stencil(w.s, w.m, Nth))


def _solver(w, node, half, ang, mode):
    import paper_1010_3816_gb300 as tk
    g = tk.Solver(rstar_min=w.rs_min, rstar_max=w.rs_max, Nr=w.Nr, Ntheta=w.Ntheta, dt=w.dt)
    tk.tk_set_coefficients(g.h, w.a, w.M, w.s, w.m, node, half, ang)
    g.set_steps_per_launch(mode)
    return g


# every number of 32-row pieces, with one column per team and with several
GRIDS = [(40, 20, 16), (40, 33, 17), (41, 97, 18), (2440, 30, 603), (2440, 30, 604), (2200, 64, 700), (1300, 128, 301)]


@pytest.mark.parametrize("Nr,Nth,c", GRIDS)
@pytest.mark.parametrize("where,q", [("node", 5), ("node", 1), ("half", 5), ("half", 6)])
def test_adjoint_next_to_a_cold_column(Nr, Nth, c, where, q):
    """One node (half node) has a large coefficient, the loss lives to its right,
    where no large term reaches: <dL, u_1> = <dL/du_0, u_0>."""
    w, node, half, ang = _tables(Nr, Nth)
    (node if where == "node" else half)[q, :, c] += LARGE
    first = c + 1 if where == "node" else c + 2
    rng = np.random.default_rng(3)
    grads = []
    for mode in (0, 1):
        g = _solver(w, node, half, ang, mode)
        for _ in range(3):
            u0 = np.zeros((4, Nth, Nr))
            u0[:, :, c - 2:first + 6] = rng.standard_normal((4, Nth, first + 8 - c))
            dL = np.zeros_like(u0)
            dL[:, :, first:first + 4] = rng.standard_normal((4, Nth, 4))
            g.set_initial(*u0)
            g.step(1)
            u1 = g.state()
            grad = np.empty_like(u0)
            g.adjoint(grad, dL_dfinal=dL, independent_pi=True)
            near = u1[:, :, first:first + 4]
            size = np.linalg.norm(dL) * np.linalg.norm(near) + np.linalg.norm(grad) * np.linalg.norm(u0)
            assert abs(np.vdot(dL, u1) - np.vdot(grad, u0)) <= TOL * size
        dL = np.random.default_rng(4).standard_normal((4, Nth, Nr))
        g.adjoint(grad, dL_dfinal=dL, independent_pi=True)
        grads.append(grad)
        g.close()
    assert np.isfinite(grads[0]).all() and np.array_equal(grads[0], grads[1])


@pytest.mark.parametrize("Nr,Nth,c", GRIDS)
@pytest.mark.parametrize("where", ["node", "half"])
def test_step_next_to_a_cold_column(Nr, Nth, c, where):
    """The forward step with a node's or a half node's coefficient made large: the
    half node and the node of that index take the FP64 instructions, so that the
    columns that use them (c and c + 1) change, those that the large coefficient
    does not enter by roundings only, and no other column changes at all."""
    w, node, half, ang = _tables(Nr, Nth)
    rng = np.random.default_rng(5)
    u0 = rng.standard_normal((4, Nth, Nr))
    out = []
    for large in (0.0, LARGE):
        (node if where == "node" else half)[5, :, c] += large
        for mode in (0, 1):
            g = _solver(w, node, half, ang, mode)
            g.set_initial(*u0)
            g.step(1)
            out.append(g.state())
            g.close()
    assert np.array_equal(out[0], out[1]) and np.array_equal(out[2], out[3])
    far = ~np.isin(np.arange(Nr), [c, c + 1])
    assert np.array_equal(out[0][:, :, far], out[2][:, :, far])
    near = np.s_[:, :, c - 1:c + 3]
    if where == "node":      # only Pi of column c has the large term
        gain = (out[2] - out[0])[2:, :, c]
        assert (np.abs(gain) > 1e3).mean() > 0.9 and np.isfinite(gain).all()
        for k in range(4):
            d = (out[2] - out[0])[k, :, c + 1 if k >= 2 else c]
            assert np.linalg.norm(d) <= TOL * np.linalg.norm(out[0][near])
