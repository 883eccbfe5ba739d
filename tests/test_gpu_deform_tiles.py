"""The warp's tile heights (32, 64 and 128 rows, by the number of tiles a launch
makes) and its two gathers (rows that share an integer displacement, and rows
that do not) give the same frame: a pair's field is bit-identical alone and in
batches large enough for the taller tiles, with predictors that are smooth, that
cross integers inside a thread's rows, and that reach outside the image."""
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


@pytest.mark.parametrize("bits", [8, 12])
@pytest.mark.parametrize("n", [8, 40])  # 64-row tiles; 128-row tiles (eager) and 64-row ones (halves of a captured batch)
@pytest.mark.parametrize("field", ["smooth", "steep", "outside"])
def test_tile_heights_and_gathers_agree(bits, n, field):
    W, H = 500, 517
    flow = synth.Flow(U=3.3, V=-1.7, vortices=[(0.5 * W, 0.5 * H, 200.0, 20.0)])
    A, B = synth.render_pair(synth.ImageSpec(W=W, H=H, bit_depth=bits, ppp=0.05, dp=(2.5, 2.5), seed=77), flow)
    a, b = rp.to_device(A), rp.to_device(B)
    eng = rp.Engine(rp.Config(W, H, windows=(16,), overlaps=(0.5,), radii=(4,), bit_depth=bits, max_batch=n))
    g = torch.Generator(device="cuda").manual_seed(5)
    y, x = torch.meshgrid(torch.arange(eng.ny, device="cuda"), torch.arange(eng.nx, device="cuda"), indexing="ij")
    if field == "smooth":
        pu, pv = 3.3 + 0.002 * x, -1.7 + 0.001 * y
    elif field == "steep":
        pu, pv = 3.3 + 2.0 * torch.randn(eng.ny, eng.nx, generator=g, device="cuda"), -1.7 + 1.5 * torch.sin(0.9 * y)
    else:
        pu, pv = 40.0 + 0.3 * y, -30.0 + 0.2 * x
    pred = (pu.float().contiguous(), pv.float().contiguous())
    ref = [t.clone() for t in eng.process_pair(a, b, pred=pred)]
    for _ in range(2):  # eager, then the captured graph
        got = eng.process_batch([a] * n, [b] * n, preds=[pred] * n)
        torch.cuda.synchronize()
        for r, t in zip(ref, got):
            assert torch.equal(t, r.expand_as(t))
    eng.close()
