"""The mixed paths' near-critical rays are traced by a kernel of their own and
skipped by the kernel of the others: every ray is traced exactly once only if
both classify alike.  The test (near_critical, csrc/tt_trace.cuh) must pick the
same rays of 64 images of 2048^2 whether the compiler contracts products into
sums or not (tests/cuda/near_critical.cu), and no pixel of an image or a batch
may be left unwritten."""
import os
import subprocess

import numpy as np
import pytest

from paper_2609_08989_gb300 import scenes

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


@pytest.fixture(scope="module")
def T():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2609_08989_gb300 import tartarus
    tartarus.lib()
    return tartarus


def test_same_rays_in_every_build(T, tmp_path):
    from paper_2609_08989_gb300 import _build
    picked = []
    for fmad in ("true", "false"):
        exe = str(tmp_path / ("near_critical_" + fmad))
        subprocess.run([_build.nvcc(), *_build.ARCH, "-std=c++17", "-O3", "-fmad=" + fmad, "-I", _build.CSRC, "-I",
                        os.path.join(ROOT, "include"), os.path.join(HERE, "cuda", "near_critical.cu"), "-o", exe],
                       check=True, capture_output=True)
        picked.append(subprocess.run([exe], check=True, capture_output=True, text=True, timeout=120).stdout.split("\n"))
    assert len(picked[0]) == 65 and picked[0] == picked[1]
    # some rays of every image, and not most of them
    assert all(0 < int(line.split()[1]) < 2048 ** 2 // 2 for line in picked[0][:64])


UNWRITTEN = -77


def poisoned(T, n):
    out = T.alloc_outputs(n)
    for v in out.values():
        v.fill_(UNWRITTEN)
    return out


@pytest.mark.parametrize("precision", [scenes.MIXED, scenes.MIXED_PAIR, scenes.MIXED_SPLIT])
def test_every_pixel_written(T, precision):
    """Codes, counts and step numbers are never negative, so a value of -77 is a
    pixel that neither kernel traced."""
    imgs = [s.replace(rtol=1e-8, atol=1e-8, critical_band=0.15)
            for s in scenes.batch_uneven(12, precision=precision, res_lo=64, res_hi=400)]
    big = scenes.kerr_disk(1024, precision).replace(rtol=1e-8, atol=1e-8, critical_band=0.15)
    ragged = big.replace(nx=611, ny=307, a=0.3, theta_obs=scenes.deg(17.0))
    for call in ([big], [ragged], imgs):
        outs = [poisoned(T, s.npix) for s in call]
        if len(call) == 1:
            T.trace(call[0], out=outs[0])
        else:
            T.trace_batch(call, outs)
        torch.cuda.synchronize()
        for sc, out in zip(call, outs):
            got = T.to_numpy(out)
            for f in ("code", "n_cross", "steps", "rejects"):
                assert not np.any(got[f] == UNWRITTEN), (sc.name, f)
