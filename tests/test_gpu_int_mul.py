"""FP64 products and conversions formed on the integer pipes (csrc/tt_soft64.cuh):
the product itself, whole step attempts that pass its range checks, and the
conversions must equal the FP64 instructions bit for bit (tests/cuda/int_mul.cu,
int_convert.cu); rays that fail the checks all the way
(an equatorial row) or a solver outside their condition (tolerances below 2^-47)
must still follow the oracle."""
import os
import subprocess

import numpy as np
import pytest

import parity
from paper_2609_08989_gb300 import scenes

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(ROOT, "paper_2609_08989_gb300", "csrc")
torch = pytest.importorskip("torch")


def _run(tmp_path, name):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2609_08989_gb300 import _build
    exe = str(tmp_path / name)
    subprocess.run([_build.nvcc(), *_build.ARCH, "-std=c++17", "-O3", "-fmad=false", "-I", CSRC, "-I",
                    os.path.join(ROOT, "include"), os.path.join(HERE, "cuda", name + ".cu"), "-o", exe],
                   check=True, capture_output=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True, timeout=120).stdout
    print(out)
    return out


def test_conversions(tmp_path):
    n, to_double, to_float, odd = _run(tmp_path, "int_convert").split()
    assert int(n) > 0 and (int(to_double), int(to_float), int(odd)) == (0, 0, 0)


def test_bits(tmp_path):
    out = _run(tmp_path, "int_mul")
    for line in out.splitlines():
        name, bad, passed, tried = line.split()
        assert int(bad) == 0, line
        # most ordinary attempts take the integer path (the odd kinds and deep stages do not)
        assert int(passed) > 0.3 * int(tried), line


@pytest.mark.parametrize("change", [dict(theta_obs=scenes.deg(90.0), nx=17, ny=9, beta_min=-9.0, beta_max=9.0),
                                    dict(nx=9, ny=8, atol=1e-15)], ids=["equatorial", "atol_below_2^-47"])
def test_outside_the_range(orc, change):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2609_08989_gb300 import tartarus as T
    sc = scenes.kerr_disk(16).replace(**change)
    out = T.trace(sc)
    torch.cuda.synchronize()
    parity.compare(orc, sc, T.to_numpy(out), orc.trace(sc), np.arange(sc.npix), rel_diverged=1e-8)
