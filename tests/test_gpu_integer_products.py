"""The FP64 sweep's products on the integer pipes have the bits of the FP64
multiplier's: 8.4 M draws of factors over every exponent, the edges of the range
checks, significands that round by ties and carries, zeros, subnormals,
infinities and NaN.  Exact, so the tolerance is zero."""
import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


def test_products_match_the_fp64_multiplier(tmp_path):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    exe = str(tmp_path / "product_check")
    src = os.path.join(HERE, "gpu_checks", "product_check.cu")
    subprocess.run([os.environ.get("NVCC", "nvcc"), "-gencode", "arch=compute_103a,code=sm_103a", "-O3",
                    "-std=c++17", "-fmad=false", "-o", exe, src], check=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split()
    assert out[0] == "mismatches" and int(out[3]) == 18 << 23
    assert int(out[1]) == 0, out
