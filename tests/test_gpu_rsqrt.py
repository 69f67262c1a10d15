"""1/sqrt of the FP64 factorisations over its range and at its branch points: a product rounded to 2^-53
enters halved, and the last sum is rounded to 2^-53; 2^-52 bounds both and the dropped 1e-22."""
import os
import subprocess

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_rsqrt(tmp_path):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2205_08417_gb300 import build
    exe = str(tmp_path / "check")
    here = os.path.dirname(os.path.abspath(__file__))
    subprocess.check_call([build._nvcc()] + build.NVCC_FLAGS + ["-o", exe, os.path.join(here, "rsqrt_check.cu")])
    worst = float(subprocess.check_output([exe]))
    print("error over 2^-52", worst)
    assert worst <= 1.0
