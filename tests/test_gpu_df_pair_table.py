"""The double-float step's sums over flows and the tabulated metric's flow, both in
packed pairs, equal the same operations one double-float at a time bit for bit
(tests/cuda/df_pair_table.cu), with and without spin."""
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
    exe = str(tmp_path_factory.mktemp("pairs") / "df_pair_table")
    subprocess.run([_build.nvcc(), *_build.ARCH, "-std=c++17", "-O3", "-I", _build.CSRC, "-I",
                    os.path.join(ROOT, "include"), os.path.join(HERE, "cuda", "df_pair_table.cu"), "-o", exe],
                   check=True, capture_output=True)
    return exe


@pytest.mark.parametrize("spin", [0.0, 0.998])
def test_bits(exe, tmp_path, spin):
    from paper_2609_08989_gb300 import tartarus as T
    nr, nth, r_min, r_max = 128, 64, 1.0 + (1.0 - spin * spin) ** 0.5, 1000.0
    coef = tmp_path / "coef.bin"
    T.table_coefficients(scenes.kerr_table_nodes(1.0, spin, nr, nth, r_min, r_max), r_min, r_max).tofile(coef)
    out = subprocess.run([exe, str(coef), str(nr), str(nth), repr(r_min), repr(r_max)], check=True,
                         capture_output=True, text=True, timeout=120).stdout
    print(out)
    lines = out.splitlines()
    assert len(lines) == 2
    for line in lines:
        name, tried, differ = line.split()
        assert int(tried) > 0 and int(differ) == 0, line
