"""How an FP32 step launches its sweeps (one launch of the three, or three), by
the launch count of a step (per stage: cell field, sweeps, update), and that the
choice does not show in the results: the bits of the same patch in a batch."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape, sweeps", [
    ((32, 32, 32), 1), ((192, 192, 1), 1), ((24, 200, 40), 1), ((1, 300, 300), 1),      # few blocks; narrow in x
    ((512, 512, 1), 3), ((384, 1, 384), 3), ((384, 384, 2), 3), ((130, 90, 100), 3),    # thin, or large
])
def test_launches(shape, sweeps):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("the expected choices are those of 152 SMs")
    from paper_1812_04278_gb300 import inputs as I, w5ct
    cons, b = I.random_smooth_state(shape, seed=8)
    dx = tuple(1.0 / n for n in shape)
    cfg = w5ct.make_config(precision=w5ct.W5CT_FP32_BULK)
    s = w5ct.Solver(shape, dx, cfg)
    s.set_state(cons, b)
    before = w5ct.w5ct_launch_count(s.ctx)
    s.step(1e-4)
    assert w5ct.w5ct_launch_count(s.ctx) - before - 1 == 4 * (2 + sweeps)   # (and dt into device memory)
    B = w5ct.Batch([shape, (8, 8, 8)], [dx, (0.125,) * 3], cfg)
    B.set_state(0, cons, b)
    B.set_state(1, *I.random_smooth_state((8, 8, 8), seed=1))
    B.step(1e-4)
    for x, y in zip(s.get_state(), B.get_state(0)):
        np.testing.assert_array_equal(x, y)
    s.close()
    B.close()
