"""The prescribed split's error norm (split_norm, csrc/tt_trace.cuh) where the FP32
flow at the new point is not finite: the attempt ends its ray with the code for a
non-finite step, as the interface promises, and is not retried
(tests/cuda/split_nan.cu)."""
import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


def test_non_finite_flow_ends_the_ray(tmp_path):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2609_08989_gb300 import _build
    exe = str(tmp_path / "split_nan")
    subprocess.run([_build.nvcc(), *_build.ARCH, "-std=c++17", "-O3", "-I", _build.CSRC, "-I",
                    os.path.join(ROOT, "include"), os.path.join(HERE, "cuda", "split_nan.cu"), "-o", exe],
                   check=True, capture_output=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True, timeout=120).stdout
    attempts, accepted, ended = (int(v) for v in out.split())
    assert ended > 0 and accepted + ended == attempts, out
