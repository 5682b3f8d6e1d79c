"""FP64 step attempts with integer products (csrc/tt_soft64.cuh) where p_phi, p_theta
or the spin is zero or tiny -- the column alpha = 0 of an image of odd width, the
equatorial plane -- and on tabulated metrics with and without spin
(tests/cuda/int_mul_zeros.cu): an attempt that passes the checks equals the plain one
bit for bit, and such states pass them (a ray that never does makes its whole warp
run both kinds of attempt)."""
import os
import subprocess

import pytest

from paper_2609_08989_gb300 import scenes

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


@pytest.fixture(scope="module")
def exe(tmp_path_factory):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2609_08989_gb300 import _build
    exe = str(tmp_path_factory.mktemp("zeros") / "int_mul_zeros")
    subprocess.run([_build.nvcc(), *_build.ARCH, "-std=c++17", "-O3", "-fmad=false", "-I", _build.CSRC, "-I",
                    os.path.join(ROOT, "include"), os.path.join(HERE, "cuda", "int_mul_zeros.cu"), "-o", exe],
                   check=True, capture_output=True)
    return exe


@pytest.mark.parametrize("spin,spherical", [(0.0, False), (0.9, False), (0.0, True)])
def test_zero_and_tiny_components(exe, tmp_path, spin, spherical):
    """spherical: a table on which g_tt, g_thth and g^rr do not vary with theta at all
    (patch coefficients of a spinless table keep rounding noise in most cells, so that
    its theta derivatives vanish only here and there)."""
    from paper_2609_08989_gb300 import tartarus as T
    nr, nth, r_min, r_max = 256, 96, 1.0 + (1.0 - spin * spin) ** 0.5, 1100.0
    coef = tmp_path / "coef.bin"
    patches = T.table_coefficients(scenes.kerr_table_nodes(1.0, spin, nr, nth, r_min, r_max), r_min, r_max)
    if spherical:
        for field in (0, 2, 4):
            patches[:, :, field, :, 1:] = 0.0
    patches.tofile(coef)
    out = subprocess.run([exe, str(coef), str(nr), str(nth), repr(r_min), repr(r_max), repr(spin)], check=True,
                         capture_output=True, text=True, timeout=120).stdout
    print(out)
    lines = out.splitlines()
    assert len(lines) == 24
    for line in lines:
        name, differ, passed, tried = line.split()
        assert int(differ) == 0, line
        # (a derivative of a table, or an error sum, may cancel to next to nothing by chance)
        assert int(passed) > 0.99 * int(tried) > 0, line
