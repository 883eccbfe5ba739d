"""The gradient of the score where the frames differ in contrast or offset (laser
pulses of unequal energy, float frames of different scales).  The score does not depend on a
gain between the frames, and every step of the adjoint is homogeneous in it: a gain
that is a power of two changes no mantissa, so the gradient keeps its bits; for any
other gain its error against 64 bits stays that of equal contrast.  Both hold for the
tiles' route and for the separate launches (128 px windows without overlap).  A
quarter is allowed between two errors, each the norm of several hundred nodes'
independent roundings (they scatter by a tenth)."""
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


def _case(W, H, w, s, seed):
    flow = synth.Flow(U=1.3, V=-0.7, vortices=[(0.5 * W, 0.5 * H, 60.0, 20.0)])
    A, B = synth.render_pair(synth.ImageSpec(W=W, H=H, bit_depth=8, ppp=0.04, dp=(2.5, 2.5), seed=seed), flow)
    nx, ny = oracle.grid_n(W, w, s), oracle.grid_n(H, w, s)
    r = synth.uniform(seed, 2 * nx * ny).reshape(2, ny, nx)
    X, Y = np.meshgrid(np.arange(nx) * s + 0.5 * (w - 1), np.arange(ny) * s + 0.5 * (w - 1))
    tu, tv = flow.eval(X, Y)
    u, v = tu + 0.4 * (r[0] - 0.5), tv + 0.4 * (r[1] - 0.5)
    return A.astype(np.float32), B.astype(np.float32), u.astype(np.float32), v.astype(np.float32)


def _gradient(A, B, w, s, u, v):
    eng = rp.Engine(rp.Config(A.shape[1], A.shape[0], windows=(w,), overlaps=(1 - s / w,), radii=(2,), float_frames=True))
    S, gu, gv = eng.score_and_grad(*[torch.from_numpy(np.ascontiguousarray(t, np.float32)).cuda() for t in (A, B, u, v)])
    out = float(S), np.stack([gu.cpu().numpy(), gv.cpu().numpy()])
    eng.close()
    return out


@pytest.mark.parametrize("W, H, w, s", [(256, 256, 32, 8), (256, 224, 16, 4), (320, 320, 64, 32), (200, 160, 16, 5),
                                        (400, 300, 128, 128)])
def test_powers_of_two_between_the_frames_change_no_bit(W, H, w, s):
    A, B, u, v = _case(W, H, w, s, 31)
    S, g = _gradient(A, B, w, s, u, v)
    for ka, kb in ((1.0, 4.0), (1.0, 256.0), (1.0 / 256.0, 1.0), (8.0, 1.0)):
        Sk, gk = _gradient(ka * A, kb * B, w, s, u, v)
        assert Sk == S and np.array_equal(gk, g), (ka, kb)


@pytest.mark.parametrize("W, H, w, s", [(256, 256, 32, 8), (256, 224, 16, 4)])
def test_error_against_64_bits_does_not_grow_with_the_gain(W, H, w, s):
    A, B, u, v = _case(W, H, w, s, 37)

    def error(a, b):
        a, b = a.astype(np.float32), b.astype(np.float32)
        _, g = _gradient(a, b, w, s, u, v)
        _, ou, ov = oracle.score_grad(a, b, w, s, u.astype(np.float64), v.astype(np.float64))
        o = np.stack([ou, ov])
        return np.linalg.norm(g - o) / np.linalg.norm(o)

    equal = error(A, B)
    for k in (3.0, 255.0):
        assert error(A, np.float32(k) * B) <= 1.25 * equal, k
    assert error(A / np.float32(3.0), B) <= 1.25 * equal
    assert error(A + np.float32(1000.0), B) <= 1.25 * equal  # an offset does not enter the score either
