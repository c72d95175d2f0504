"""The div b maximum is that of the cells without a NaN, wherever the NaN lies:
in the first cell of a block, in a cell whose thread also has the largest
value, or in the last cell.  Against numpy on the same faces (three differences
and two sums of O(1) numbers times 1/dx: 1e-13 relative)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SHAPE = (64, 64, 96)
STRIDE = 1024 * 256          # threads of the reduction


@pytest.mark.parametrize("bad", [0, 256 * 5, 100000, 64 * 64 * 96 - 1])
@pytest.mark.parametrize("top", [3, 256 * 5 + 40, 100000 + STRIDE, 20000])
def test_maximum(bad, top):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1812_04278_gb300 import inputs as I, w5ct
    cons, b = I.random_smooth_state(SHAPE, seed=4)
    b[1].reshape(-1)[top] += 0.25
    b[2].reshape(-1)[bad] = np.nan
    dx = tuple(1.0 / n for n in SHAPE)
    div = sum((b[d] - np.roll(b[d], 1, axis=2 - d)) / dx[d] for d in range(3))
    s = w5ct.Solver(SHAPE, dx)
    s.set_state(cons, b)
    np.testing.assert_allclose(s.div_b_norm()[0], np.nanmax(np.abs(div)), rtol=1e-13)
    s.close()
