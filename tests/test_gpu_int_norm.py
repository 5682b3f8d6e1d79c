"""The error norm with integer products over the tolerances that a solver may ask
for: equal to the plain one bit for bit wherever its checks pass
(tests/cuda/int_norm.cu), and an absolute tolerance next to zero, which leaves the
relative one alone, does not send the whole step back to plain products."""
import os
import subprocess

import pytest

from paper_2609_08989_gb300 import scenes

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


def test_bits_over_the_tolerances(tmp_path):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2609_08989_gb300 import _build
    exe = str(tmp_path / "int_norm")
    subprocess.run([_build.nvcc(), *_build.ARCH, "-std=c++17", "-O3", "-fmad=false", "-I", _build.CSRC, "-I",
                    os.path.join(ROOT, "include"), os.path.join(HERE, "cuda", "int_norm.cu"), "-o", exe],
                   check=True, capture_output=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True, timeout=120).stdout
    print(out)
    for line in out.splitlines():
        rtol, atol, differ, passed, tried = (float(v) for v in line.split())
        assert differ == 0, line
        # seven of eight states have a theta and p_theta away from zero: their factors,
        # rtol |y| + atol with |y| in e^-5 .. e^7, have products within 2^+-200
        if 1e-27 <= max(rtol, atol) <= 2.0 ** 47:
            assert passed >= 0.875 * tried, line


def test_small_absolute_tolerance_is_as_fast():
    """atol just above and far below 2^-47 at rtol 1e-10: the same step attempts
    within 2 %, plain products take 1.9 times as long."""
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2609_08989_gb300 import tartarus as T
    best = {}
    for atol in (7.2e-15, 1e-15, 1e-30):
        sc = scenes.kerr_disk(384).replace(atol=atol)
        out = T.alloc_outputs(sc.npix)
        T.trace(sc, out=out)
        ms = []
        for _ in range(5):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record()
            T.trace(sc, out=out)
            b.record()
            torch.cuda.synchronize()
            ms.append(a.elapsed_time(b))
        best[atol] = min(ms) / (out["steps"].sum().item() + out["rejects"].sum().item())
    assert best[1e-15] < 1.3 * best[7.2e-15] and best[1e-30] < 1.3 * best[7.2e-15], best
