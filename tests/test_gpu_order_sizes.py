"""The order from the middle of the image (csrc/tt_trace.cuh tile_pixel) is taken by
launches of more than 256 rays per SM on the FP64, double-float, tabulated and
prescribed-split paths: sized from the device, every pixel of such a launch is traced
exactly once, whole images and ranges, single and in a batch."""
import numpy as np
import pytest

from paper_2609_08989_gb300 import scenes

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

FIELDS = ("code", "n_cross", "r_cross", "g", "I_cross", "intensity", "steps", "rejects")
PATHS = {"fp64": scenes.FP64, "double_float": scenes.DOUBLE_FLOAT, "split": scenes.MIXED_SPLIT,
         "table_fp64": scenes.FP64, "table_double_float": scenes.DOUBLE_FLOAT}


@pytest.fixture(scope="module")
def T():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2609_08989_gb300 import tartarus
    tartarus.lib()
    return tartarus


def threshold():
    return 256 * torch.cuda.get_device_properties(0).multi_processor_count


def scene(path, nx, ny, **kw):
    base = scenes.table_kerr_with_nodes(16) if path.startswith("table") else scenes.kerr_disk(16)
    return base.replace(precision=PATHS[path], nx=nx, ny=ny, rtol=1e-6, atol=1e-6, alpha_min=-12.0, alpha_max=12.0, **kw)


def poisoned(T, n):
    out = T.alloc_outputs(n)
    for v in out.values():
        v.fill_(-77)
    return out


@pytest.mark.parametrize("path", sorted(PATHS))
@pytest.mark.parametrize("nx,beta", [(208, (-12.0, 12.0)), (211, (-12.0, 12.0)), (208, (2.0, 14.0))])
def test_every_pixel_once(T, path, nx, beta):
    rows = (threshold() * 21 // 20 // nx + 4) // 4 * 4
    sc = scene(path, nx, rows + 8, beta_min=beta[0], beta_max=beta[1])
    table = T.Table(sc.table, sc.r_min, sc.r_max) if path.startswith("table") else None
    begin, count = (4 * nx, rows * nx) if nx % 8 == 0 else (3 * nx + 5, rows * nx + 7)
    assert count > threshold()
    got = T.to_numpy(T.trace(sc, out=poisoned(T, count), table=table, pix_begin=begin, pix_count=count))
    # the same range in parts that keep the order of beta
    step = nx * (threshold() // (2 * nx))
    parts = [T.to_numpy(T.trace(sc, table=table, pix_begin=p, pix_count=min(step, begin + count - p)))
             for p in range(begin, begin + count, step)]
    for f in FIELDS:
        assert np.array_equal(got[f], np.concatenate([p[f] for p in parts], axis=-1)), f


@pytest.mark.parametrize("path", ["fp64", "double_float", "split"])
def test_batch(T, path):
    side = int((threshold() / 4) ** 0.5)
    imgs = [scene(path, side + 16 * k, side + 9 * k, beta_min=-12.0 + 3 * k, beta_max=12.0, a=0.9 - 0.2 * k)
            for k in range(4)]
    assert sum(s.npix for s in imgs) > threshold() and all(s.npix <= threshold() for s in imgs)
    outs = [poisoned(T, s.npix) for s in imgs]
    T.trace_batch(imgs, outs)
    torch.cuda.synchronize()
    for sc, out in zip(imgs, outs):
        got = T.to_numpy(out)
        for f in ("code", "n_cross", "steps", "rejects"):
            assert not np.any(got[f] == -77), f
        if path == "fp64":                  # every width of the FP64 kernel rounds alike
            ref = T.to_numpy(T.trace(sc))
            for f in FIELDS:
                assert np.array_equal(got[f], ref[f]), f
