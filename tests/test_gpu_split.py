"""The FP64 step's integer coupling (csrc/tk_split.cuh) and its transpose
(csrc/tk_split_adjoint.cuh): teams of warps at the edges of their 32-row pieces
and of the radial split, all launch structures on the same bits, powers of two
of the data, and the columns that take the FP64 instructions (huge values,
infinities).

Tolerances.  With the oracle's own coefficients a run differs from the oracle
by roundings only: per Lax-Wendroff step a value takes at most 16 of them
(2^-53 each, on terms of at most the size of the field next to it) on either
side, so after n steps of fields that do not grow by more than a factor of ten
the relative L2 distance stays below 10 * 2 * 16 * n * 2^-53; n = 6 gives 2.2e-13.
"""
import math

import numpy as np
import pytest

from inputs import Workload, initial_planes

pytestmark = pytest.mark.gpu

N = 6
TOL = 10 * 2 * 16 * N * 2.0 ** -53


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_1010_3816_gb300 as tk
    tk.load_library()


def _work(Nr, Nth, **kw):
    drs = 1.0 / 8.0
    rs_min = -2.0
    # the innermost and outermost rows and columns an observer may name, and
    # rows on both sides of a 32-row edge
    th = [(j + 0.75) * math.pi / Nth for j in {0, min(31, Nth - 2), Nth - 2}]
    obs = tuple((rs_min + (Nr - 1) * drs * f, t) for f, t in zip((0.0, 0.5, 1.0), th))
    base = dict(name="split", a=0.9, m=2, rs_min=rs_min, rs_max=rs_min + (Nr - 1) * drs, Nr=Nr, Ntheta=Nth,
                dt=1 / 64, center=rs_min + 0.4 * (Nr - 1) * drs, width=2.0, noise=1e-3, seed=11, observers=obs)
    base.update(kw)
    return Workload(**base)


def _solver(w, mode=0, coeffs=None):
    import paper_1010_3816_gb300 as tk
    g = tk.Solver(rstar_min=w.rs_min, rstar_max=w.rs_max, Nr=w.Nr, Ntheta=w.Ntheta, dt=w.dt, substeps=w.substeps,
                  variable=w.variable)
    if coeffs is None:
        g.precompute(w.a, w.M, w.s, w.m)
    else:
        tk.tk_set_coefficients(g.h, w.a, w.M, w.s, w.m, *coeffs)
    g.set_steps_per_launch(mode)
    return g


def _run(w, mode=0, scale=1.0, n=N, coeffs=None):
    g = _solver(w, mode, coeffs)
    re, im = initial_planes(w)
    g.set_initial(re * scale, im * scale)
    ids = [g.add_observer(r, t) for r, t in w.observers]
    g.step(n)
    out = g.state(), [g.waveform(k) for k in ids]
    g.close()
    return out


def _oracle(w, n=N):
    """The oracle's run and its coefficients as tk_set_coefficients takes them
    (its half nodes are stored one column to the right)."""
    import oracle
    o = oracle.Solver(M=w.M, a=w.a, s=w.s, m=w.m, rs_min=w.rs_min, rs_max=w.rs_max, Nr=w.Nr, Ntheta=w.Ntheta,
                      dt=w.dt, substeps=w.substeps, variable=w.variable)
    ids = [o.add_observer(r, t) for r, t in w.observers]
    o.set_initial(*initial_planes(w))
    node, half = o.coeffs()
    half9 = np.zeros_like(half)
    half9[:, :, :-1] = half[:, :, 1:]
    ang = np.stack(oracle.regular_stencil(w.s, w.m, w.Ntheta)) if w.variable else None
    o.run(n)
    return (o.state(), [o.waveform(k) for k in ids]), (node, half9, ang)


SIZES = [(3, 2), (5, 31), (17, 32), (40, 33), (153, 63), (700, 64), (333, 65), (90, 97), (1300, 128), (2440, 30)]


@pytest.mark.parametrize("Nr,Nth", SIZES)
@pytest.mark.parametrize("kind", ["kerr", "schwarzschild", "literal"])
def test_edges_against_the_oracle(Nr, Nth, kind):
    kw = {"kerr": {}, "schwarzschild": dict(a=0.0, m=1), "literal": dict(variable=0, s=0, m=1, dt=1 / 512)}[kind]
    w = _work(Nr, Nth, **kw)
    (ref, wref), coeffs = _oracle(w)
    got, wgot = _run(w, coeffs=coeffs)
    for c in range(4):
        assert np.linalg.norm(got[c] - ref[c]) <= TOL * np.linalg.norm(ref[c]), c
    for a, b in zip(wgot, wref):
        assert np.linalg.norm(a - b) <= TOL * max(np.linalg.norm(x) for x in wref)


@pytest.mark.parametrize("Nr,Nth,scale", [(700, 64, 1.0), (333, 97, 1.0), (90, 40, 2.0 ** 880), (153, 20, 2.0 ** 876)])
def test_launch_structures_agree(Nr, Nth, scale):
    """One persistent launch, one launch per step, pairs of steps and a batch:
    the same bits, also where columns are cold (values above 2^877)."""
    import paper_1010_3816_gb300 as tk
    w = _work(Nr, Nth, substeps=2)
    ref, wref = _run(w, -1, scale)
    assert np.isfinite(ref).all()
    for mode in (1, 2):
        s, wv = _run(w, mode, scale)
        assert np.array_equal(s, ref) and all(np.array_equal(a, b) for a, b in zip(wv, wref)), mode
    gs = [_solver(w), _solver(w)]
    re, im = initial_planes(w)
    for g in gs:
        g.set_initial(re * scale, im * scale)
        for r, t in w.observers:
            g.add_observer(r, t)
    b = tk.Batch(gs)
    b.step(N)
    for g in gs:
        assert np.array_equal(g.state(), ref)
        assert all(np.array_equal(g.waveform(k), v) for k, v in enumerate(wref))
    b.close()


@pytest.mark.parametrize("p", [-700, -3, 500])
def test_powers_of_two_scale_exactly(p):
    """The step is linear and every value carries its own exponent, so a power
    of two passes through to the bit."""
    w = _work(200, 64)
    s1, w1 = _run(w)
    s2, w2 = _run(w, scale=2.0 ** p)
    assert np.array_equal(s2, s1 * 2.0 ** p)
    assert all(np.array_equal(b, a * 2.0 ** p) for a, b in zip(w1, w2))


@pytest.mark.parametrize("p", [870, 877, 890])
def test_cold_columns_agree_with_the_others(p):
    """Above 2^877 a column takes the FP64 instructions: the same result but for
    its roundings."""
    w = _work(200, 64)
    s1, _ = _run(w)
    s2, _ = _run(w, scale=2.0 ** p)
    s2 = s2 * 2.0 ** -p
    for c in range(4):
        assert np.linalg.norm(s2[c] - s1[c]) <= TOL * np.linalg.norm(s1[c])


@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan])
@pytest.mark.parametrize("Nth,j,comp", [(64, 31, 0), (97, 64, 1), (20, 0, 2), (128, 127, 3)])
def test_a_non_finite_value_stays_in_its_stencil(bad, Nth, j, comp):
    """One step spreads it to the columns next to it and two rows each way (one
    per half step), and nowhere else; the state is then reported unstable."""
    import paper_1010_3816_gb300 as tk
    w = _work(80, Nth)
    i = 37
    g = _solver(w)
    g.set_initial(*initial_planes(w))
    s0 = g.state()
    g.step(1)
    ref = g.state()
    s0[comp, j, i] = bad
    g.set_state(s0)
    g.step(1)
    s1 = g.state()
    hit = ~np.isfinite(s1)
    assert hit[:, j, i].any()
    rows, cols = np.nonzero(hit.any(axis=0))
    assert (abs(cols - i) <= 1).all() and (abs(rows - j) <= 2).all()
    far = np.abs(np.arange(w.Nr) - i) > 1
    assert np.array_equal(s1[:, :, far], ref[:, :, far])
    near = ~hit & ~far[None, None, :]
    assert np.abs(s1 - ref)[near & (np.abs(np.arange(Nth) - j) > 2)[None, :, None]].max() <= \
        16 * 2.0 ** -53 * 10 * np.abs(ref).max()
    with pytest.raises(tk.TkError):
        g.check_finite()
    g.close()


# ---- the transposed step (csrc/tk_split_adjoint.cuh) ----

def _adjoint(w, mode=0, scale=1.0, n=3):
    """(initial planes, final state, its loss gradient, dL/d(initial planes))."""
    g = _solver(w, mode)
    rng = np.random.default_rng(5)
    u0 = rng.standard_normal((4, w.Ntheta, w.Nr))
    u0[:, :, [0, -1]] = 0.0
    g.set_initial(*u0)
    g.step(n)
    dL = rng.standard_normal(u0.shape)
    dL[:, :, [0, -1]] = 0.0
    grad = np.empty_like(u0)
    g.adjoint(grad, dL_dfinal=dL * scale, independent_pi=True)
    uN = g.state()
    g.close()
    return u0, uN, dL * scale, grad


@pytest.mark.parametrize("Nr,Nth", SIZES)
@pytest.mark.parametrize("a", [0.9, 0.0])
def test_adjoint_is_the_transpose_at_the_edges(Nr, Nth, a):
    """<dL, u_N> = <dL/du_0, u_0>: each side is off by the roundings of three
    steps, 16 of 2^-53 each, times the growth allowed above."""
    u0, uN, dL, grad = _adjoint(_work(Nr, Nth, a=a))
    norm = np.linalg.norm
    assert abs(np.vdot(dL, uN) - np.vdot(grad, u0)) <= TOL * (norm(dL) * norm(uN) + norm(grad) * norm(u0))


@pytest.mark.parametrize("Nr,Nth,scale", [(700, 64, 1.0), (333, 97, 1.0), (90, 40, 2.0 ** 877), (153, 20, 2.0 ** 890)])
def test_adjoint_launch_structures_agree(Nr, Nth, scale):
    """One persistent launch and one launch per step: the same bits, also where
    columns are cold, and there the others' result but for its roundings."""
    w = _work(Nr, Nth, substeps=2)
    ref = _adjoint(w, -1, scale)[3]
    assert np.isfinite(ref).all()
    assert np.array_equal(_adjoint(w, 1, scale)[3], ref)
    plain = _adjoint(w)[3]
    assert np.linalg.norm(ref / scale - plain) <= TOL * np.linalg.norm(plain)


@pytest.mark.parametrize("p", [-700, 500])
def test_adjoint_powers_of_two_scale_exactly(p):
    w = _work(200, 64)
    assert np.array_equal(_adjoint(w, scale=2.0 ** p)[3], _adjoint(w)[3] * 2.0 ** p)


def test_adjoint_tables_follow_the_coefficients():
    """A solver precomputed again uses the new black hole's tables."""
    w = _work(90, 40)
    g = _solver(w)
    rng = np.random.default_rng(6)
    u0 = rng.standard_normal((4, w.Ntheta, w.Nr))
    dL = rng.standard_normal(u0.shape)
    grads = []
    for a in (0.9, 0.3):
        g.precompute(a, w.M, w.s, w.m)
        g.set_initial(*u0)
        g.step(2)
        grads.append(np.empty_like(u0))
        g.adjoint(grads[-1], dL_dfinal=dL, independent_pi=True)
    g.close()
    h = _solver(w.with_(a=0.3))
    h.set_initial(*u0)
    h.step(2)
    want = np.empty_like(u0)
    h.adjoint(want, dL_dfinal=dL, independent_pi=True)
    h.close()
    assert np.array_equal(grads[1], want) and not np.array_equal(grads[0], want)


@pytest.mark.parametrize("Nr,Nth", [(9, 20), (130, 45), (333, 97), (1700, 32)])
def test_param_gradient_does_not_depend_on_the_grouping(Nr, Nth):
    """The transposed steps are contracted up to eight at a time, at most those
    of a checkpoint interval: every grouping gives the same bits, and one step
    at a time (C = substeps = 1) is the plain order."""
    for k in (1, 3):
        w = _work(Nr, Nth, substeps=k)
        g = _solver(w)
        g.set_initial(*initial_planes(w))
        g.add_observer(w.rs_min + 0.6 * (Nr - 1) * w.drs, 1.1)
        g.step(11)
        dL = np.random.default_rng(7).standard_normal((1, 11, 2))
        grads = [g.param_gradient("a", dL, C) for C in (1, 0, 4, 11)]
        g.close()
        assert np.isfinite(grads[0]) and grads[0] != 0.0
        assert grads == [grads[0]] * 4


@pytest.mark.parametrize("Nr,Nth", [(4, 32), (1824, 20), (1825, 32), (2128, 32), (2129, 32), (912, 64), (913, 50),
                                    (1064, 64), (1065, 64), (456, 128), (457, 97)])
def test_small_grid_launch_at_its_edges(Nr, Nth):
    """One column per team, at the ends of its range and of its blocks of three
    or seven columns: the bits of one launch per step, state and samples, for an
    odd number of steps too."""
    w = _work(Nr, Nth, substeps=1)
    for n in (2, 5):
        ref, wref = _run(w, 1, n=n)
        s, wv = _run(w, 0, n=n)
        assert np.array_equal(s, ref) and all(np.array_equal(a, b) for a, b in zip(wv, wref))


@pytest.mark.parametrize("Nr,Nth,k", [(4, 32, 1), (5, 20, 2), (1824, 32, 1), (1825, 32, 1), (911, 50, 3), (912, 64, 1),
                                      (913, 64, 1), (455, 128, 2), (456, 97, 1), (457, 128, 1)])
def test_small_grid_adjoint_at_its_edges(Nr, Nth, k):
    """The transposed step with one column per team, at the ends of its range and
    of its blocks of three: the bits of one launch per step."""
    w = _work(Nr, Nth, substeps=k)
    assert np.array_equal(_adjoint(w, 0)[3], _adjoint(w, 1)[3])
