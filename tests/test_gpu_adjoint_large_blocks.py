"""Score and gradient with blocks above 32 px, whose moments eight warps share: the
smallest such block, sizes that are no multiple of a warp or of the eight warps' stride,
the largest, and windows of one and of several of them.  Tolerances as for the smaller
blocks (2e-4 of the gradient's norm, 1e-5 of the score)."""
import numpy as np
import pytest
import torch

import oracle
import paper_2504_17987_gb300 as rp
import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2504_17987_gb300 import build
    build.build()
    oracle.build()
    synth.build()


@pytest.mark.parametrize("W, H, w, s", [(150, 141, 34, 34), (260, 210, 100, 50), (231, 160, 66, 33), (300, 300, 96, 96),
                                        (400, 270, 126, 42), (520, 270, 128, 128)])
def test_score_and_gradient_match_the_oracle(W, H, w, s):
    flow = synth.Flow(U=1.3, V=-0.7, vortices=[(0.5 * W, 0.5 * H, 60.0, 20.0)])
    A, B = synth.render_pair(synth.ImageSpec(W=W, H=H, bit_depth=12, ppp=0.05, dp=(2.5, 2.5), seed=23), flow)
    nx, ny = oracle.grid_n(W, w, s), oracle.grid_n(H, w, s)
    r = synth.uniform(29, 2 * nx * ny).reshape(2, ny, nx)
    u, v = (1.3 + 0.4 * (r[0] - 0.5)).astype(np.float32), (-0.7 + 0.4 * (r[1] - 0.5)).astype(np.float32)
    eng = rp.Engine(rp.Config(W, H, windows=(w,), overlaps=(1 - s / w,), radii=(2,), bit_depth=12))
    S, gu, gv = eng.score_and_grad(rp.to_device(A), rp.to_device(B), torch.from_numpy(u).cuda(), torch.from_numpy(v).cuda())
    So, ou, ov = oracle.score_grad(A, B, w, s, u.astype(np.float64), v.astype(np.float64))
    assert abs(float(S) - So) <= 1e-5 * abs(So)
    g, o = np.stack([gu.cpu().numpy(), gv.cpu().numpy()]), np.stack([ou, ov])
    assert np.linalg.norm(g - o) <= 2e-4 * np.linalg.norm(o)
    eng.close()
