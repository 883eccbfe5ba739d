"""Captured batches of host frames run in parts whose uploads overlap the passes of
the parts before: their fields equal a device-frames engine's captured batch bit for
bit, at part counts of 1 to 4 and in both halves of a split batch, with schedules
whose strips depend on the number of pairs, and on the eager first call."""
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


@pytest.mark.parametrize("n", [1, 2, 3, 5, 17])
@pytest.mark.parametrize("windows,radii,levels", [((32, 16), (4, 4), 1), ((64, 16), (4, 1), 0)])
def test_parts_equal_the_uncut_batch(n, windows, radii, levels):
    W, H = 3341, 630  # 3341-byte rows start anywhere in a 16-byte word; 4.2 MB per pair: one pair per part and more
    flow = synth.Flow(U=1.3, V=-0.7, vortices=[(0.5 * W, 0.5 * H, 200.0, 20.0)])
    base = synth.render_pair(synth.ImageSpec(W=W, H=H, bit_depth=8, ppp=0.02, dp=(2.5, 2.5), seed=300), flow)
    pairs = [(np.roll(base[0], 7 * k, 0), np.roll(base[1], 7 * k, 0)) for k in range(n)]
    kw = dict(windows=windows, overlaps=(0.5,) * len(windows), radii=radii, levels=levels, max_batch=n)
    dev, host = rp.Engine(rp.Config(W, H, **kw)), rp.Engine(rp.Config(W, H, host_frames=True, **kw))
    da, db = [rp.to_device(p[0]) for p in pairs], [rp.to_device(p[1]) for p in pairs]
    ha, hb = ([rp.to_device(p[k], "cpu", pin=True) for p in pairs] for k in (0, 1))
    for _ in range(3):  # eager, then captured
        ref, got = dev.process_batch(da, db), host.process_batch(ha, hb)
        torch.cuda.synchronize()
        for x, y in zip(ref, got):
            assert torch.equal(x, y)
    host.wait(10000)
    dev.close()
    host.close()


@pytest.mark.parametrize("shift", [0, 1, 3])
def test_predictors_in_other_pairs_outputs_are_read_before_they_are_written(shift):
    """Every pair's predictor is the output memory of another pair (or, shift 0, its own):
    the fields equal those of a call whose predictors lie elsewhere."""
    W, H, n = 3341, 630, 4
    flow = synth.Flow(U=1.3, V=-0.7, vortices=[(0.5 * W, 0.5 * H, 200.0, 20.0)])
    base = synth.render_pair(synth.ImageSpec(W=W, H=H, bit_depth=8, ppp=0.02, dp=(2.5, 2.5), seed=301), flow)
    ha, hb = ([rp.to_device(np.roll(base[k], 7 * i, 0), "cpu", pin=True) for i in range(n)] for k in (0, 1))
    eng = rp.Engine(rp.Config(W, H, windows=(16,), overlaps=(0.5,), radii=(2,), max_batch=n, host_frames=True))
    fields = [[torch.full((eng.ny, eng.nx), 0.9 + 0.1 * i + 0.05 * k, device="cuda") for k in (0, 1)] for i in range(n)]
    ref = eng.process_batch(ha, hb, preds=[tuple(f) for f in fields])
    torch.cuda.synchronize()
    for _ in range(3):  # eager, then captured
        outs = eng.empty_outputs(n)
        for i in range(n):
            outs[0][i], outs[1][i] = fields[i]
        preds = [(outs[0][(i + n - shift) % n], outs[1][(i + n - shift) % n]) for i in range(n)]
        want = ref if not shift else eng.process_batch(ha, hb, preds=[tuple(fields[(i + n - shift) % n]) for i in range(n)])
        got = eng.process_batch(ha, hb, preds=preds, outs=outs)
        torch.cuda.synchronize()
        for x, y in zip(want, got):
            assert torch.equal(x, y)
    eng.wait(10000)
    eng.close()


@pytest.mark.parametrize("bits", [8, 12])
@pytest.mark.parametrize("W", [64, 255, 256, 257, 530, 1029])
@pytest.mark.parametrize("offset", [0, 1, 3, 13])
def test_upload_of_rows_at_any_alignment(bits, W, offset):
    """Rows that start anywhere in a 16-byte word, ragged ends, rows of one to several
    warps: the fields equal those of the same frames on the device."""
    H = 72
    flow = synth.Flow(U=1.3, V=-0.7, vortices=[])
    A, B = synth.render_pair(synth.ImageSpec(W=W, H=H, bit_depth=bits, ppp=0.05, dp=(2.5, 2.5), seed=W), flow)
    kw = dict(windows=(16,), overlaps=(0.5,), radii=(2,), bit_depth=bits)
    dev, host = rp.Engine(rp.Config(W, H, **kw)), rp.Engine(rp.Config(W, H, host_frames=True, **kw))
    views = []
    for img in (A, B):
        t = rp.to_device(img, "cpu", pin=False)
        buf = torch.zeros(H, W + offset + 2, dtype=t.dtype).pin_memory()
        buf[:, offset:offset + W] = t
        views.append(buf[:, offset:offset + W])
    ref, got = dev.process_pair(rp.to_device(A), rp.to_device(B)), host.process_pair(*views)
    torch.cuda.synchronize()
    for x, y in zip(ref, got):
        assert torch.equal(x, y)
    dev.close()
    host.close()
