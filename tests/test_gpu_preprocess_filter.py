"""The high-pass filter alone (no equalisation), whose chunks are the frame's own (128
columns, 16 rows): sizes around a chunk's edges, the largest box, and a result that does
not depend on the histogram tiles.  The filtered value is an exact integer over the
box's pixel count, so one float division away from the oracle's (1e-6 vmax)."""
import numpy as np
import pytest
import torch

import oracle
import paper_2504_17987_gb300 as rp

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2504_17987_gb300 import build
    build.build()
    oracle.build()


@pytest.mark.parametrize("W,H,dtype,vmax,hp", [(1, 1, np.uint8, 255, 3), (128, 16, np.uint8, 255, 64), (129, 17, np.uint16, 4095, 64),
                                               (127, 15, np.uint8, 255, 0), (391, 277, np.uint8, 255, 64),
                                               (700, 33, np.uint16, 65535, 7), (3, 500, np.uint16, 4095, 5)])
def test_filter_alone(W, H, dtype, vmax, hp):
    rng = np.random.default_rng(11 * W + H)
    img = rng.integers(0, min(65536, vmax + 1) if dtype == np.uint16 else 256, (H, W)).astype(dtype)
    t = rp.to_device(img)
    out = rp.stage_preprocess(t, vmax, hp=hp, tiles=(1, 1), clip_pct=0)
    ref = oracle.preprocess(img.astype(np.float64), vmax, hp=hp, tiles=(1, 1), clip_pct=0)
    assert np.abs(out.cpu().numpy().astype(np.float64) - ref).max() <= 1e-6 * vmax
    tiles = (min(W, 64), min(H, 64))
    assert torch.equal(rp.stage_preprocess(t, vmax, hp=hp, tiles=tiles, clip_pct=0), out)
