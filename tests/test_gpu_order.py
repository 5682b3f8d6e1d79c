"""The order in which queue entries are handed out (csrc/tt_trace.cuh tile_pixel):
every pixel of a range is traced exactly once, whatever the range's shape and
wherever the line beta = 0 lies, so a range's outputs equal those of the same
pixels in the whole image."""
import numpy as np
import pytest

from paper_2609_08989_gb300 import scenes

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

# (nx, ny, first pixel, pixels or 0 for the rest): tiles, one tile row, ragged
# runs, less than one run, a last part of a run; beta = 0 inside, above, below
RANGES = [(16, 12, 0, 0), (8, 4, 0, 0), (16, 24, 64, 128), (9, 7, 0, 0), (5, 3, 2, 9), (33, 11, 40, 300), (40, 1, 0, 0),
          (240, 168, 0, 0), (241, 165, 7, 0)]       # more rays than lanes: outward from the middle


@pytest.mark.parametrize("precision", [scenes.FP64, scenes.DOUBLE_FLOAT, scenes.MIXED_PAIR])
@pytest.mark.parametrize("beta", [(-6.0, 6.0), (1.0, 9.0), (-9.0, -1.0), (3.0, 3.0)])
def test_every_pixel_once(precision, beta):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2609_08989_gb300 import tartarus as T
    for nx, ny, begin, count in RANGES:
        sc = scenes.kerr_disk(16, precision).replace(nx=nx, ny=ny, beta_min=beta[0], beta_max=beta[1], rtol=1e-8,
                                                     atol=1e-8)
        # the whole image band by band (row by row when small): each call one range
        # with an order of its own
        band = nx * max(1, ny // 12)
        rows = [T.to_numpy(T.trace(sc, pix_begin=p, pix_count=min(band, nx * ny - p)))
                for p in range(0, nx * ny, band)]
        n = count or nx * ny - begin
        out = T.alloc_outputs(n)
        for v in out.values():
            v.fill_(-77)
        got = T.to_numpy(T.trace(sc, out=out, pix_begin=begin, pix_count=n))
        for f in ("code", "n_cross", "r_cross", "g", "intensity", "steps", "rejects"):
            ref = np.concatenate([r[f] for r in rows], axis=-1)[..., begin:begin + n]
            assert np.array_equal(got[f], ref), (f, nx, ny, begin, count)
