"""Score and gradient where the adjoint's work is cut: blocks of 1 to 32 px and
above (64 px windows without overlap), node tiles at the image's edge, grids of a
single row or column, images wider than the windows' union, and repeated calls on
one handle (the score's ticket).  The tolerance (2e-4 of the gradient's norm, 1e-5
of the score) is the one the full-size test derives for FP32 sums of this length."""
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


@pytest.mark.parametrize("W,H,w,overlap,bits", [
    (64, 48, 16, 0.75, 8),      # 4 px blocks
    (101, 87, 16, 0.6875, 8),   # steps of 5 px: blocks of one pixel
    (40, 36, 8, 0.875, 8),      # steps of one pixel
    (90, 77, 24, 0.5, 12),      # 12 px blocks, a border the windows do not reach
    (32 + 10, 200, 32, 0.5, 8),  # one column of nodes
    (300, 45, 32, 0.75, 12),    # two rows of nodes
    (170, 201, 64, 0.5, 8),     # 32 px blocks, node tiles of two by one
    (210, 140, 64, 0.0, 12),    # 64 px blocks
    (300, 280, 128, 0.0, 8),    # 128 px blocks: node tiles that do not fit
])
def test_score_and_gradient_where_the_work_is_cut(W, H, w, overlap, bits):
    s = int(round(w * (1 - overlap)))
    flow = synth.Flow(U=1.3, V=-0.7, vortices=[(0.5 * W, 0.5 * H, 60.0, 20.0)])
    A, B = synth.render_pair(synth.ImageSpec(W=W, H=H, bit_depth=bits, ppp=0.05, dp=(2.5, 2.5), seed=17), flow)
    nx, ny = oracle.grid_n(W, w, s), oracle.grid_n(H, w, s)
    r = synth.uniform(19, 2 * nx * ny).reshape(2, ny, nx)
    u, v = (1.3 + 0.4 * (r[0] - 0.5)).astype(np.float32), (-0.7 + 0.4 * (r[1] - 0.5)).astype(np.float32)
    eng = rp.Engine(rp.Config(W, H, windows=(w,), overlaps=(overlap,), radii=(2,), bit_depth=bits))
    args = rp.to_device(A), rp.to_device(B), torch.from_numpy(u).cuda(), torch.from_numpy(v).cuda()
    S, gu, gv = eng.score_and_grad(*args)
    So, ou, ov = oracle.score_grad(A, B, w, s, u.astype(np.float64), v.astype(np.float64))
    assert abs(float(S) - So) <= 1e-5 * abs(So)
    g, o = np.stack([gu.cpu().numpy(), gv.cpu().numpy()]), np.stack([ou, ov])
    assert np.linalg.norm(g - o) <= 2e-4 * np.linalg.norm(o)
    again = [eng.score_and_grad(*args, want_grad=False)[0] for _ in range(3)]
    assert all(torch.equal(t, S) for t in again)
    eng.close()
