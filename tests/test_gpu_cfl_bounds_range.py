"""The float bounds of speed_kernel's double CFL maxima hold over the whole
range of units.  Against the oracle's maxima, 1e-13 relative (the parity bar of
one evaluation): a cell whose squared speeds overflow float when squared once
more must not shadow the others (overflow), and states whose speeds are so
small that their fourth powers underflow must keep a bound above the speed
(small).  Several iterations of a warp, so that published maxima are read."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SHAPE = (128, 128, 96)


def check(rho, v, P, B):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import oracle
    from paper_1812_04278_gb300 import inputs as I, w5ct
    b = np.stack([np.full(rho.shape, x) for x in B])
    cons, b = I.assemble(rho, v, P, b, Bc=b.copy())
    dx = tuple(1.0 / m for m in SHAPE)
    o = oracle.Oracle(SHAPE, dx, oracle.make_config())
    o.set_state(cons, b)
    s = w5ct.Solver(SHAPE, dx, w5ct.make_config())
    s.set_state(cons, b)
    np.testing.assert_allclose(s.max_signal_speed(), o.max_signal_speed(), rtol=1e-13)
    s.close()


# speeds of the shadowing cell and of the fastest one; the fastest in the same
# warp, and in a later iteration of the same warp (8 x 152 blocks of 256)
@pytest.mark.parametrize("pressure, velocity", [(3e19, 2e10), (1.3e19, 1e10), (1e25, 1e13), (1e29, 1e15)])
@pytest.mark.parametrize("at", [5, 3 * 8 * 152 * 256 + 17])
def test_overflow(pressure, velocity, at):
    n = SHAPE[::-1]
    rho, P, v = np.ones(n), np.full(n, pressure / 300.0), np.zeros((3,) + n)
    P.reshape(-1)[0] = pressure
    for d in range(3):
        v[d].reshape(-1)[at + 8 * d] = velocity
    check(rho, v, P, (0.0, 0.0, 0.0))


# speeds within 30% of one another, the scale of their squares from 1e-26 to 1e34
@pytest.mark.parametrize("exponent", range(-26, 35, 5))
@pytest.mark.parametrize("field", [0.0, 0.7])
def test_small(exponent, field):
    n = SHAPE[::-1]
    rng = np.random.default_rng(exponent + 100)
    scale = 10.0 ** exponent
    v = rng.uniform(-0.3, 0.3, (3,) + n) * scale ** 0.5
    P = scale * rng.uniform(1.0, 1.2, n)
    check(np.ones(n), v, P, tuple(field * scale ** 0.5 * w for w in (0.6, 0.5, -0.4)))


# the pressure alone sets the speed, and one cell of the last iteration wins by 10%
@pytest.mark.parametrize("exponent", [-26, -24, -22, -20])
def test_small_winner(exponent):
    n = SHAPE[::-1]
    P = np.full(n, 10.0 ** exponent)
    P.reshape(-1)[-100] *= 1.21
    check(np.ones(n), np.zeros((3,) + n), P, (0.0, 0.0, 0.0))
