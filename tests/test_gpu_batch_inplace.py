"""A batch large enough to be captured in parts (16 pairs and more), every pair's
predictor in the output memory of another pair or its own, device and host frames:
the fields equal those of a call whose predictors lie elsewhere, bit for bit, on the
eager first call and on the captured ones."""
import numpy as np
import pytest
import torch

import paper_2504_17987_gb300 as rp
import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2504_17987_gb300 import build
    build.build()
    synth.build()


@pytest.mark.parametrize("host", [False, True])
@pytest.mark.parametrize("n, shift", [(16, 0), (16, 8), (17, 9), (17, 16), (33, 17)])
def test_fields_handed_on_in_place(n, shift, host):
    W, H = 640, 480
    flow = synth.Flow(U=1.3, V=-0.7, vortices=[(0.5 * W, 0.5 * H, 60.0, 20.0)])
    base = synth.render_pair(synth.ImageSpec(W=W, H=H, bit_depth=8, ppp=0.03, dp=(2.5, 2.5), seed=302), flow)
    where = dict(device="cpu", pin=True) if host else {}
    a, b = ([rp.to_device(np.roll(base[k], 7 * i, 0), **where) for i in range(n)] for k in (0, 1))
    eng = rp.Engine(rp.Config(W, H, windows=(16,), overlaps=(0.5,), radii=(2,), max_batch=n, host_frames=host))
    fields = [[torch.full((eng.ny, eng.nx), 0.9 + 0.02 * i + 0.05 * k, device="cuda") for k in (0, 1)] for i in range(n)]
    src = [(i + shift) % n for i in range(n)]
    for _ in range(2):  # both patterns eager, then captured
        want = eng.process_batch(a, b, preds=[tuple(fields[j]) for j in src])
    for _ in range(3):
        outs = eng.empty_outputs(n)
        for i in range(n):
            outs[0][i], outs[1][i] = fields[i]
        got = eng.process_batch(a, b, preds=[(outs[0][j], outs[1][j]) for j in src], outs=outs)
        torch.cuda.synchronize()
        for x, y in zip(want, got):
            assert torch.equal(x, y)
    eng.wait(10000)
    eng.close()
