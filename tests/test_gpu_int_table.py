"""Direct tests of what the FP64 table path and the step control compute in place of
library operations (tests/cuda/int_table.cu): division by a constant from its
reciprocal, a table's cell index from the bits of a coordinate (last cell, values
below 0 and beyond 2^21, infinities, NaN), the next step size.  Built as the FP64
kernels are and, with contraction, as the prescribed split's kernel is; step
attempts with integer products equal plain ones in the latter build too."""
import os
import subprocess

import pytest

from paper_2609_08989_gb300 import scenes

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


def build(tmp_path, name, fmad):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2609_08989_gb300 import _build
    exe = str(tmp_path / name)
    subprocess.run([_build.nvcc(), *_build.ARCH, "-std=c++17", "-O3", "-fmad=" + fmad, "-I", _build.CSRC, "-I",
                    os.path.join(ROOT, "include"), os.path.join(HERE, "cuda", name + ".cu"), "-o", exe],
                   check=True, capture_output=True)
    return exe


@pytest.mark.parametrize("fmad", ["false", "true"])
def test_division_cell_and_next_step(tmp_path, fmad):
    out = subprocess.run([build(tmp_path, "int_table", fmad)], check=True, capture_output=True, text=True,
                         timeout=120).stdout
    print(out)
    lines = out.splitlines()
    assert len(lines) == 3
    for line in lines:
        name, tried, differ = line.split()
        assert int(tried) > 0 and int(differ) == 0, line


def test_step_attempts_with_contraction(tmp_path):
    from paper_2609_08989_gb300 import tartarus as T
    exe = build(tmp_path, "int_mul_zeros", "true")
    nr, nth, spin, r_max = 256, 96, 0.9, 1100.0
    r_min = 1.0 + (1.0 - spin * spin) ** 0.5
    coef = tmp_path / "coef.bin"
    T.table_coefficients(scenes.kerr_table_nodes(1.0, spin, nr, nth, r_min, r_max), r_min, r_max).tofile(coef)
    out = subprocess.run([exe, str(coef), str(nr), str(nth), repr(r_min), repr(r_max), repr(spin)], check=True,
                         capture_output=True, text=True, timeout=120).stdout
    print(out)
    for line in out.splitlines():
        name, differ, passed, tried = line.split()
        assert int(differ) == 0 and int(passed) > 0, line
