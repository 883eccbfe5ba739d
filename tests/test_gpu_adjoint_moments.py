"""The windows' moments, formed from their blocks' (up to 32 x 32 blocks here): the
score against 64 bits to one FP32 unit, 2^-24.  Each coefficient carries the rounding
of its moments, a few units of either sign, and the score is the sum of a hundred and
more of them: their average lies well inside one unit, unless the roundings of the
moments lean to one side."""
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


@pytest.mark.parametrize("W, H, w, s, ppp", [(640, 640, 64, 32, 0.04), (256, 240, 64, 6, 0.04), (480, 400, 64, 16, 0.004),
                                             (333, 277, 16, 5, 0.01)])
def test_the_score_stays_within_one_unit(W, H, w, s, ppp):
    flow = synth.Flow(U=1.3, V=-0.7, vortices=[(0.5 * W, 0.5 * H, 60.0, 20.0)])
    A, B = synth.render_pair(synth.ImageSpec(W=W, H=H, bit_depth=8, ppp=ppp, dp=(2.5, 2.5), seed=53), flow)
    nx, ny = oracle.grid_n(W, w, s), oracle.grid_n(H, w, s)
    X, Y = np.meshgrid(np.arange(nx) * s + 0.5 * (w - 1), np.arange(ny) * s + 0.5 * (w - 1))
    u, v = [t.astype(np.float32) for t in flow.eval(X, Y)]
    eng = rp.Engine(rp.Config(W, H, windows=(w,), overlaps=(1 - s / w,), radii=(2,)))
    S = eng.score_and_grad(rp.to_device(A), rp.to_device(B), torch.from_numpy(u).cuda(), torch.from_numpy(v).cuda(),
                           want_grad=False)[0]
    So = oracle.score_grad(A, B, w, s, u.astype(np.float64), v.astype(np.float64), grad=False)
    eng.close()
    assert abs(float(S) - So) <= 2.0 ** -24 * abs(So)


@pytest.mark.parametrize("seed", [100, 200])
def test_a_background_does_not_take_the_means_digits(seed):
    """Sparse particles, half of them lost, on a background of 100 to 102 counts.  A
    block's mean rounds once to FP32, by 2.2e-6 counts on average; sixteen blocks make a
    window, and the noise its terms are measured against has 0.8 counts: about 0.7e-6 of
    the gradient.  A sum of 64 pixels in the digits of 6400 rounds as much once more
    (1e-6 together), and once per addition: 1.1e-6 is allowed."""
    W = H = 256
    w, s = 32, 8
    rng = np.random.default_rng(seed)
    n = int(0.003 * W * H)
    x, y, amp = rng.uniform(0, W, n), rng.uniform(0, H, n), rng.uniform(100, 1000, n)
    keep = rng.uniform(size=n) > 0.5
    yy, xx = np.mgrid[0:H, 0:W]

    def frame(px, py, a):
        img = np.zeros((H, W))
        for X, Y, q in zip(px, py, a):
            i0, i1, j0, j1 = max(0, int(X) - 5), min(W, int(X) + 6), max(0, int(Y) - 5), min(H, int(Y) + 6)
            if i1 > i0 and j1 > j0:
                img[j0:j1, i0:i1] += q * np.exp(-((xx[j0:j1, i0:i1] - X) ** 2 + (yy[j0:j1, i0:i1] - Y) ** 2) / 1.5)
        return np.round(img + 100 + rng.integers(0, 3, (H, W))).astype(np.float32)

    A, B = frame(x, y, amp), frame(x[keep] + 1.3, y[keep] - 0.7, amp[keep])
    nx, ny = oracle.grid_n(W, w, s), oracle.grid_n(H, w, s)
    u = (1.3 + 0.4 * rng.uniform(-0.5, 0.5, (ny, nx))).astype(np.float32)
    v = (-0.7 + 0.4 * rng.uniform(-0.5, 0.5, (ny, nx))).astype(np.float32)
    eng = rp.Engine(rp.Config(W, H, windows=(w,), overlaps=(0.75,), radii=(2,), float_frames=True))
    _, gu, gv = eng.score_and_grad(*[torch.from_numpy(t).cuda() for t in (A, B, u, v)])
    _, ou, ov = oracle.score_grad(A, B, w, s, u.astype(np.float64), v.astype(np.float64))
    eng.close()
    g, o = np.stack([gu.cpu().numpy(), gv.cpu().numpy()]), np.stack([ou, ov])
    assert np.linalg.norm(g - o) <= 1.1e-6 * np.linalg.norm(o)
