"""The FP64 face arithmetic's helpers and its rare branches on the GPU.

* The reciprocal square root and division of the FP64 sweep (one third-order
  step from the hardware's approximation) against the correctly rounded
  values on 16.7 M arguments: each ends in one FMA whose result carries the
  rounding of its small correction and of one product, so at most 2 units in
  the last place; the exact helpers (power-of-two scaling, comparisons on the
  bit patterns) must agree everywhere.
* Appendix A's fallback a_f = a_s = 1 at c_f = c_slow exactly, where the left
  and right eigenvectors are not inverses and the central flux goes through
  both: every interface along x of the first stage meets it.
"""
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module", autouse=True)
def cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def test_rsqrt_and_division_within_two_ulps(tmp_path):
    exe = str(tmp_path / "rsqrt_check")
    src = os.path.join(HERE, "gpu_checks", "rsqrt_check.cu")
    subprocess.run([os.environ.get("NVCC", "nvcc"), "-gencode", "arch=compute_103a,code=sm_103a", "-O3",
                    "-std=c++17", "-o", exe, src], check=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split()
    assert int(out[7]) == 1 << 24
    assert int(out[1]) <= 2 and int(out[3]) <= 2 and int(out[5]) == 0, out


@pytest.mark.parametrize("variant", [0, 1])
def test_triple_point_fallback_matches_oracle(variant):
    """gamma = 2, P = 1/2, rho = 1, B = (1, 0, 0): c_s = c_A exactly and
    B_t = 0; dyadic velocities along x keep P exact in the recovery, so the
    first stage's x-faces all take the fallback.  One step of dt = 1e-5
    against the oracle: the bar is the parity bar, 1e-12 of the state scale.
    (At dt = 1e-5 a central flux left unprojected would be off by O(dt/dx)
    = 1e-4.)"""
    import oracle
    from paper_1812_04278_gb300 import w5ct
    shape, dx = (16, 8, 8), (1.0 / 16, 1.0 / 8, 1.0 / 8)
    i = np.arange(16)
    vx = np.broadcast_to(((i * 5) % 16) / 64.0, (8, 8, 16)).copy()
    cons = np.zeros((5, 8, 8, 16))
    cons[0] = 1.0
    cons[1] = vx
    cons[4] = 0.5 + 0.5 * vx * vx + 0.5
    bface = np.zeros((3, 8, 8, 16))
    bface[0] = 1.0
    o = oracle.Oracle(shape, dx, oracle.make_config(weno_variant=variant, gamma=2.0))
    o.set_state(cons, bface)
    s = w5ct.Solver(shape, dx, w5ct.make_config(weno_variant=variant, gamma=2.0))
    s.set_state(cons, bface)
    o.step(1e-5)
    s.step(1e-5)
    oc, ob, _ = o.get_state()
    gc, gb, _ = s.get_state()
    scale = max(np.abs(oc).max(), np.abs(ob).max())
    assert max(np.abs(gc - oc).max(), np.abs(gb - ob).max()) <= 1e-12 * scale
    assert np.abs(gc - cons).max() > 1e-6
    s.close()
