"""Float frames and pyramid levels made in one launch: level 1 of every format at
sizes around the kernel's 4 x 4 patches, and engines with one to four levels (two
per launch) whose fields must equal those of frames with an unaligned row pitch
(single loads instead of vector ones) bit for bit."""
import numpy as np
import pytest
import torch

import paper_2504_17987_gb300 as rp
import synth
from paper_2504_17987_gb300 import binding

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2504_17987_gb300 import build
    build.build()
    synth.build()


@pytest.mark.parametrize("dtype", [np.uint8, np.uint16, np.float32])
@pytest.mark.parametrize("W,H", [(2, 2), (3, 5), (4, 4), (7, 6), (9, 3), (127, 33), (128, 34), (130, 35), (515, 70)])
def test_level_one_is_the_box_mean(W, H, dtype):
    rng = np.random.default_rng(W * H)
    img = rng.integers(0, 200, (H, W)).astype(dtype)
    t = torch.from_numpy(img).cuda() if dtype == np.float32 else rp.to_device(img)
    e = img[: H // 2 * 2, : W // 2 * 2].astype(np.float64)
    ref = (e[0::2, 0::2] + e[0::2, 1::2] + e[1::2, 0::2] + e[1::2, 1::2]) / 4  # exact in FP32
    got = binding.stage_downsample(t).cpu().numpy()
    assert np.array_equal(got, ref.astype(np.float32))


@pytest.mark.parametrize("levels", [1, 2, 3, 4])
@pytest.mark.parametrize("deform", ["b", "central"])
def test_levels_do_not_depend_on_the_load_form(levels, deform):
    W, H = 701, 666  # odd levels on the way down
    flow = synth.Flow(U=6.3, V=-2.7, vortices=[(0.5 * W, 0.5 * H, 200.0, 20.0)])
    A, B = synth.render_pair(synth.ImageSpec(W=W, H=H, bit_depth=12, ppp=0.05, dp=(2.5, 2.5), seed=91), flow)
    cfg = rp.Config(W, H, windows=(16,), overlaps=(0.5,), radii=(4,), levels=levels, bit_depth=12, deform=deform)
    eng = rp.Engine(cfg)
    outs = []
    for pad in (703, 704):  # rows of 1406 bytes: single loads; 1408: vector loads
        dev = []
        for img in (A, B):
            buf = torch.zeros(H, pad, dtype=torch.int16, device="cuda")
            buf[:, :W] = rp.to_device(img)
            dev.append(buf[:, :W])
        outs.append([t.clone() for t in eng.process_pair(*dev)])
    torch.cuda.synchronize()
    for x, y in zip(*outs):
        assert torch.equal(x, y)
    eng.close()
