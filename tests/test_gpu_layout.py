"""The transposes between the planes [Ntheta][Nr] and the device state, in tiles of
32 rows by 8 or 32 columns: both directions exact at the tiles' edges and on both
sides of the line between the two, and the derived momentum to the bit, with the
spacing a power of two (a multiplication there) and not."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SIZES = [(5, 16), (33, 33), (40, 128), (9727, 20), (9728, 32), (4864, 45), (2431, 128), (2432, 97)]


def _solver(Nr, Nth, drs, precision=0):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_1010_3816_gb300 as tk
    g = tk.Solver(rstar_min=-1.0, rstar_max=-1.0 + (Nr - 1) * drs, Nr=Nr, Ntheta=Nth, dt=1 / 1024,
                  precision=precision)
    g.precompute(0.9, 1.0, -2, 2)
    return g


@pytest.mark.parametrize("Nr,Nth", SIZES)
@pytest.mark.parametrize("precision", [0, 1])
def test_state_round_trip(Nr, Nth, precision):
    g = _solver(Nr, Nth, 0.25, precision)
    u = np.random.default_rng(1).standard_normal((4, Nth, Nr))
    g.set_initial(u[0], u[1])
    g.set_state(u)
    want = (u.astype(np.float32) if precision else u).astype(np.float64)
    want[:, :, [0, -1]] = 0.0
    assert np.array_equal(g.state(), want)
    g.set_initial(*u)
    assert np.array_equal(g.state(), want)
    g.close()


@pytest.mark.parametrize("Nr,Nth", SIZES)
@pytest.mark.parametrize("drs", [0.25, 0.3])
def test_derived_momentum(Nr, Nth, drs):
    import paper_1010_3816_gb300 as tk
    g = _solver(Nr, Nth, drs)
    u = np.random.default_rng(2).standard_normal((2, Nth, Nr))
    g.set_initial(u[0], u[1])
    b = tk.tk_get_coefficients(g.h, (Nth, Nr))[0][0]
    spacing = ((-1.0 + (Nr - 1) * drs) - -1.0) / (Nr - 1)
    got = g.state()[2:, :, 1:-1]
    g.close()
    assert np.array_equal(got, b[:, 1:-1] * (u[:, :, 2:] - u[:, :, :-2]) / (2.0 * spacing))
