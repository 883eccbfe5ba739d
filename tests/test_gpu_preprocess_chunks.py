"""Pre-processing where its work is cut: chunks of a histogram tile (16 rows, 512
columns), staged strips (256 columns), runs of four pixels, rows of eight, tiles
smaller than a chunk, tiles past the image, the largest box and pixels above vmax.
The tolerance (1e-4 vmax) admits float rounding of the maps and the blend only: a
wrong bin or count shows as an error of the order of vmax / 256."""
import numpy as np
import pytest

import oracle
import paper_2504_17987_gb300 as rp

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2504_17987_gb300 import build
    build.build()
    oracle.build()


@pytest.mark.parametrize("W,H,dtype,vmax,hp,tiles,clip", [
    (1, 1, np.uint8, 255, 0, (1, 1), 200),
    (1, 1, np.uint16, 65535, 64, (1, 1), 200),
    (513, 33, np.uint16, 4095, 64, (1, 1), 200),   # two chunk columns, two chunk rows
    (257, 31, np.uint8, 255, 1, (1, 1), 200),      # one past a staged strip, one short of two chunk rows
    (1100, 17, np.uint16, 65535, 7, (1, 2), 300),  # three chunk columns, strips inside them
    (65, 70, np.uint8, 255, 7, (64, 64), 200),     # tiles of two pixels, half of them past the image
    (3, 900, np.uint16, 4095, 2, (1, 1), 100),     # narrow: chunks of at least 512 pixels
    (130, 47, np.uint8, 100, 3, (3, 2), 150),      # pixels above vmax fall in the last bin
    (255, 19, np.uint16, 4095, 9, (2, 1), 0),      # the filter alone
])
def test_preprocess_where_the_work_is_cut(W, H, dtype, vmax, hp, tiles, clip):
    rng = np.random.default_rng(7 * W + H)
    top = 256 if dtype == np.uint8 else min(65536, vmax + 1)
    img = rng.integers(0, top, (H, W)).astype(dtype)
    img[: (H + 1) // 2] //= 16  # a dark half: a peaked histogram that clipping acts on
    out = rp.stage_preprocess(rp.to_device(img), vmax, hp=hp, tiles=tiles, clip_pct=clip).cpu().numpy()
    ref = oracle.preprocess(img.astype(np.float64), vmax, hp=hp, tiles=tiles, clip_pct=clip)
    assert np.abs(out.astype(np.float64) - ref).max() <= 1e-4 * vmax
