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
