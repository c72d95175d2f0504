"""The double CFL maxima skip cells whose float bounds rule them out
(speed_kernel): the result must be the maximum over every cell all the same.
Against the oracle's maxima on states where the bounds are tight, useless or
misleading: uniform (every cell ties), one cell that wins by 1e-9 of the
maximum (below float's resolution), pressures that are small differences of
the energy, floors, values beyond float's range, and grids whose cell count
is not a multiple of a warp.  The bar is the parity bar of one evaluation,
1e-13 relative."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(5, 3, 7), (33, 9, 10), (64, 48, 40)])
@pytest.mark.parametrize("kind", ["smooth", "uniform", "winner", "cold", "floored", "huge"])
def test_maxima_are_those_of_every_cell(shape, kind):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import oracle
    from paper_1812_04278_gb300 import inputs as I, w5ct
    rng = np.random.default_rng(3)
    n = shape[::-1]
    if kind == "smooth":
        cons, b = I.random_smooth_state(shape, seed=5)
    else:
        cons, b = I.uniform_state(shape, v=(0.3, -0.2, 0.1), B=(0.5, 0.4, -0.3))
    if kind == "winner":
        at = tuple(rng.integers(0, m) for m in n)
        cons[(1,) + at] *= 1.0 + 1e-9
        cons[(4,) + at] += 0.5 * (cons[(1,) + at] ** 2 - 0.3 ** 2)
    if kind in ("cold", "floored"):
        # kinetic energy 1e6 times the thermal one (and, floored, none at all in places)
        cons[1:4] = rng.normal(size=(3,) + n) * 30.0
        cons[4] = 0.5 * (cons[1:4] ** 2).sum(0) + 0.25 + rng.uniform(0.001, 0.002, n)
        if kind == "floored":
            cons[4] -= 0.05 * (rng.random(n) < 0.3)
    if kind == "huge":
        cons, b = cons * 1e60, b * 1e30
    floors = int(kind == "floored")
    dx = tuple(1.0 / m for m in shape)
    o = oracle.Oracle(shape, dx, oracle.make_config(floors=floors, rho_min=1e-3, p_min=1e-3))
    o.set_state(cons, b)
    s = w5ct.Solver(shape, dx, w5ct.make_config(floors=floors, rho_min=1e-3, p_min=1e-3))
    s.set_state(cons, b)
    np.testing.assert_allclose(s.max_signal_speed(), o.max_signal_speed(), rtol=1e-13)
    s.close()
