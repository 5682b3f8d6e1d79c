"""The double-float flow in packed pairs equals the one by component bit for bit
(tests/cuda/df_pairs.cu), with and without spin, outside and just inside the
horizon, for angles beyond (0, pi)."""
import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


def test_bits(tmp_path):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2609_08989_gb300 import _build
    exe = str(tmp_path / "df_pairs")
    subprocess.run([_build.nvcc(), *_build.ARCH, "-std=c++17", "-O3", "-I", _build.CSRC, "-I",
                    os.path.join(ROOT, "include"), os.path.join(HERE, "cuda", "df_pairs.cu"), "-o", exe],
                   check=True, capture_output=True)
    states, differ = subprocess.run([exe], check=True, capture_output=True, text=True, timeout=120).stdout.split()
    assert int(states) > 0 and int(differ) == 0
