"""What the FP64 step's integer coupling and its transpose owe to the FP64
instructions they replace, value by value and not in the norm of a plane: every
theta row to its own size, both signs alike, correct rounding, gradual underflow.

The reference is the step of Eqs. (lw1) and (lw2) term by term in numpy's
longdouble, with the solver's raw coefficients.  The bound of a result is the same
sum over the absolute values of its terms, B: an entry of the tables and a stage
(half node, node) of FP64 operations each cost at most 24 roundings of 2^-53 of the
terms they join, so that |got - exact| <= 64 2^-53 B.
"""
import numpy as np
import pytest

from inputs import Workload

pytestmark = pytest.mark.gpu

TOL = 64 * 2.0 ** -53
LD = np.longdouble


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_1010_3816_gb300 as tk
    tk.load_library()


def _work(Nr, Nth, rs_min=-2.0, drs=1 / 8, **kw):
    base = dict(name="acc", a=0.9, m=2, rs_min=rs_min, rs_max=rs_min + (Nr - 1) * drs, Nr=Nr, Ntheta=Nth, dt=1 / 64)
    base.update(kw)
    return Workload(**base)


def _solver(w, mode=0):
    import paper_1010_3816_gb300 as tk
    g = tk.Solver(rstar_min=w.rs_min, rstar_max=w.rs_max, Nr=w.Nr, Ntheta=w.Ntheta, dt=w.dt)
    g.precompute(w.a, w.M, w.s, w.m)
    g.set_steps_per_launch(mode)
    return g


class Exact:
    """The regularised step from raw coefficients: lists of terms (out, in, side,
    row offset, coefficient), out and in of Phi_R, Phi_I, Pi_R, Pi_I."""

    def __init__(self, w, node, half, ang):
        self.Nr = w.Nr
        drs = LD(w.rs_max - w.rs_min) / (w.Nr - 1)
        self.half = self._terms(half[:, :, :-1].astype(LD), ang.astype(LD), LD(w.dt) / 2, drs, True)
        self.node = self._terms(node[:, :, 1:-1].astype(LD), ang.astype(LD), LD(w.dt), drs, False)

    @staticmethod
    def _terms(raw, ang, tau, drs, average):
        b, c1, c2, c3, c4 = raw[0], (raw[1], raw[2]), (raw[3], raw[4]), (raw[5], raw[6]), raw[7]
        up, dn = c4 * ang[0][:, None], c4 * ang[1][:, None]
        half = LD(1) / 2
        t = []
        for side, sg in ((0, -1), (1, 1)):
            d = sg * tau / drs
            for p in range(2):
                if average:
                    t += [(p, p, side, 0, half + 0 * b), (2 + p, 2 + p, side, 0, half + 0 * b)]
                t += [(p, p, side, 0, -d * b), (p, 2 + p, side, 0, tau * half + 0 * b), (2 + p, 2 + p, side, 0, d * b),
                      (2 + p, p, side, 0, -tau * half * (up + dn)), (2 + p, p, side, 1, tau * half * up),
                      (2 + p, p, side, -1, tau * half * dn)]
                for q in range(2):     # (x + iy)(u + iv)
                    z = (lambda c: c[0] if p == q else (c[1] if p == 1 else -c[1]))
                    t += [(2 + p, q, side, 0, d * z(c1)), (2 + p, q, side, 0, tau * half * z(c3)),
                          (2 + p, 2 + q, side, 0, tau * half * z(c2))]
        return t

    @staticmethod
    def _rows(x, dj):     # x[j + dj], zero beyond the grid
        y = np.zeros_like(x)
        if dj == 0:
            y[:] = x
        elif dj > 0:
            y[:-1] = x[1:]
        else:
            y[1:] = x[:-1]
        return y

    def step(self, u, f=lambda c: c):
        n = self.Nr
        h = np.zeros((4,) + (u.shape[1], n - 1), LD)
        for o, i, side, dj, c in self.half:
            h[o] += f(c) * self._rows(u[i], dj)[:, side:side + n - 1]
        new = np.zeros(u.shape, LD)
        new[:, :, 1:-1] = u[:, :, 1:-1]
        for o, i, side, dj, c in self.node:
            new[o][:, 1:-1] += f(c) * self._rows(h[i], dj)[:, side:side + n - 2]
        return new

    def transpose(self, v, f=lambda c: c):
        n = self.Nr
        v = v.copy()
        v[:, :, [0, -1]] = 0
        h = np.zeros((4,) + (v.shape[1], n - 1), LD)
        for o, i, side, dj, c in self.node:
            h[i][:, side:side + n - 2] += self._rows(f(c) * v[o][:, 1:-1], -dj)
        g = v
        for o, i, side, dj, c in self.half:
            g[i][:, side:side + n - 1] += self._rows(f(c) * h[o], -dj)
        g[:, :, [0, -1]] = 0     # the edges' initial data are not used
        return g


def _case(w, mode):
    """A solver and its exact step, both on the oracle's coefficients."""
    import oracle
    import paper_1010_3816_gb300 as tk
    o = oracle.Solver(M=w.M, a=w.a, s=w.s, m=w.m, rs_min=w.rs_min, rs_max=w.rs_max, Nr=w.Nr, Ntheta=w.Ntheta, dt=w.dt)
    node, h = o.coeffs()
    half = np.zeros_like(h)
    half[:, :, :-1] = h[:, :, 1:]
    ang = np.stack(oracle.regular_stencil(w.s, w.m, w.Ntheta))
    g = tk.Solver(rstar_min=w.rs_min, rstar_max=w.rs_max, Nr=w.Nr, Ntheta=w.Ntheta, dt=w.dt)
    tk.tk_set_coefficients(g.h, w.a, w.M, w.s, w.m, node, half, ang)
    g.set_steps_per_launch(mode)
    return g, Exact(w, node, half, ang)


def _check(got, exact, bound):
    bad = np.abs(got.astype(LD) - exact) > TOL * bound
    assert not bad.any(), [tuple(int(v) for v in k) + (float(abs(got[tuple(k)] - exact[tuple(k)]) / bound[tuple(k)]),)
                           for k in np.argwhere(bad)[:5]]


def _transpose(g, w, dL, n=1):
    g.set_initial(*np.zeros((4, w.Ntheta, w.Nr)))
    g.step(n)
    grad = np.empty(dL.shape)
    g.adjoint(grad, dL_dfinal=dL, independent_pi=True)
    return grad


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("Nth", [30, 64, 97])
@pytest.mark.parametrize("s,m", [(-2, 4), (-2, 16), (-2, 32), (0, 32), (-2, 64), (0, 0)])
def test_adjoint_rows_next_to_the_poles(s, m, Nth, mode):
    """The adjoint state of the regularised field goes with the weight of its cell,
    which next to a pole changes by many powers of two from row to row, and the
    neighbours' coefficients by as many the other way."""
    import oracle
    w = _work(9, Nth, s=s, m=m)
    th = (np.arange(Nth) + 0.5) * (np.pi / Nth)
    weight = np.array([np.sin(t) * oracle.weight(s, m, 1, t) ** 2 for t in th])[None, :, None]
    dL = weight * (1.0 + 0.5 * np.random.default_rng(1).standard_normal((4, Nth, w.Nr)))
    dL[:, :, [0, -1]] = 0.0
    g, E = _case(w, mode)
    grad = _transpose(g, w, dL)
    g.close()
    _check(grad, E.transpose(dL.astype(LD)), E.transpose(np.abs(dL).astype(LD), np.abs))


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("Nth", [30, 64, 97])
@pytest.mark.parametrize("kw", [dict(), dict(a=0.0), dict(s=0, m=8), dict(rs_min=-300.0), dict(rs_min=-300.0, s=0, m=0),
                                dict(rs_min=-1000.0, drs=1.0), dict(rs_min=500.0, drs=1.0, m=12)])
@pytest.mark.parametrize("spread", [4, 40, 400])
def test_neighbours_of_very_different_size(kw, Nth, mode, spread):
    """Every value with an exponent of its own, the step and its transpose; also
    close to the horizon, where the neighbours' coefficients vanish, and far out."""
    w = _work(9, Nth, **kw)
    rng = np.random.default_rng(spread)
    shape = (4, Nth, w.Nr)
    u, dL = (rng.standard_normal(shape) * 2.0 ** rng.integers(-spread, spread + 1, shape) for _ in range(2))
    u[:, :, [0, -1]] = dL[:, :, [0, -1]] = 0.0
    g, E = _case(w, mode)
    grad = _transpose(g, w, dL)
    g.set_initial(*u)
    g.step(1)
    got = g.state()
    g.close()
    _check(got, E.step(u.astype(LD)), E.step(np.abs(u).astype(LD), np.abs))
    _check(grad, E.transpose(dL.astype(LD)), E.transpose(np.abs(dL).astype(LD), np.abs))


# every number of 32-row pieces, with one column per team and with several
SIZES = [(60, 20), (60, 50), (60, 97), (2300, 30), (2200, 64), (1300, 128)]


@pytest.mark.parametrize("Nr,Nth", SIZES)
@pytest.mark.parametrize("mode", [0, 1])
def test_both_signs_alike(Nr, Nth, mode):
    """The step of -u and the gradient of -dL are the negatives of those of u and
    dL to the bit, with neighbours of very different size."""
    w = _work(Nr, Nth)
    rng = np.random.default_rng(2)
    shape = (4, Nth, Nr)
    u0, dL = (rng.standard_normal(shape) * 2.0 ** rng.integers(-30, 30, shape) for _ in range(2))
    g = _solver(w, mode)
    out = []
    for sign in (1.0, -1.0):
        g.set_initial(*(sign * u0))
        g.step(3)
        grad = np.empty(shape)
        g.adjoint(grad, dL_dfinal=sign * dL, independent_pi=True)
        out.append((g.state(), grad))
    g.close()
    assert np.array_equal(out[0][0], -out[1][0])
    assert np.array_equal(out[0][1], -out[1][1])


@pytest.mark.parametrize("Nr,Nth", SIZES)
@pytest.mark.parametrize("mode", [0, 1])
def test_representable_couplings_are_exact(Nr, Nth, mode):
    """With c3 alone and Phi = 1 the new Pi is dt c3, a number of 53 bits, and
    the transpose of a single Pi = 1 gives Phi such numbers (its Pi, 1 + dt^2 c3 / 4,
    is none): nothing but the rounding of the integer sum to FP64 can change a bit."""
    import paper_1010_3816_gb300 as tk
    w = _work(Nr, Nth)
    rng = np.random.default_rng(9)
    node, half = np.zeros((2, 9, Nth, Nr))
    node[5:7] = rng.standard_normal((2, Nth, Nr))
    g = tk.Solver(rstar_min=w.rs_min, rstar_max=w.rs_max, Nr=w.Nr, Ntheta=w.Ntheta, dt=w.dt)
    tk.tk_set_coefficients(g.h, w.a, w.M, w.s, w.m, node, half, np.zeros((2, Nth)))
    g.set_steps_per_launch(mode)
    E = Exact(w, node, half, np.zeros((2, Nth)))
    u = np.zeros((4, Nth, Nr))
    u[0, :, 1:-1] = 1.0
    dL = np.zeros_like(u)
    dL[2, :, 2:-2:4] = 1.0
    grad = _transpose(g, w, dL)
    g.set_initial(*u)
    g.step(1)
    got = g.state()
    g.close()
    inner = np.s_[:, :, 2:-2]      # (next to the edges Phi's half nodes are 1/2)
    want = E.step(u.astype(LD))
    assert np.array_equal(got[inner], want[inner].astype(float))
    assert np.array_equal(np.abs(got[2][:, 2:-2]), np.abs(w.dt * node[5][:, 2:-2]))
    assert np.array_equal(grad[:2], E.transpose(dL.astype(LD))[:2].astype(float))


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("Nth", [30, 64, 97])
@pytest.mark.parametrize("p", [-960, -1010, -1040, -1060])
@pytest.mark.parametrize("kw", [dict(), dict(s=0, m=0, rs_min=-1440.0)])
def test_gradual_underflow(kw, p, Nth, mode):
    """Tiny data: each of at most 64 roundings costs 2^-1075 at least, and 4 / dt as
    much in the Phi that the transposed half nodes keep times dt / 4 (near the horizon
    the neighbours' coefficients are subnormal too)."""
    w = _work(9, Nth, **kw)
    rng = np.random.default_rng(-p)
    shape = (4, Nth, w.Nr)
    u, dL = (rng.standard_normal(shape) * 2.0 ** p for _ in range(2))
    u[:, :, [0, -1]] = dL[:, :, [0, -1]] = 0.0
    g, E = _case(w, mode)
    grad = _transpose(g, w, dL)
    g.set_initial(*u)
    g.step(1)
    got = g.state()
    g.close()
    floor = 64 * 4 / w.dt * LD(2.0) ** -1075 / TOL
    _check(got, E.step(u.astype(LD)), E.step(np.abs(u).astype(LD), np.abs) + floor)
    _check(grad, E.transpose(dL.astype(LD)), E.transpose(np.abs(dL).astype(LD), np.abs) + floor)
