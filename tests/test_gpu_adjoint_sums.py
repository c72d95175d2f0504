"""The adjoint step's sums over faces keep more than float in either arithmetic
type (double, or pairs of floats): face adjoints of 2^30 that cancel leave the
small integers beside them exact (the sums are integers below 2^33, their
result below 2^24: no rounding at all, so the tolerance is zero)."""
import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


def test_cancelling_sums_are_exact(tmp_path):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    exe = str(tmp_path / "adj_sum_check")
    src = os.path.join(HERE, "gpu_checks", "adj_sum_check.cu")
    subprocess.run([os.environ.get("NVCC", "nvcc"), "-gencode", "arch=compute_103a,code=sm_103a", "-O2",
                    "-std=c++17", "-o", exe, src], check=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split()
    assert [float(x) for x in out[1:4] + out[5:8]] == [0.0] * 6, out
