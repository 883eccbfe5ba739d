"""The pass kernels specialised to 50 % overlap (blocks of 8, 12, 16, 24 and 32 px,
radii 1 to 8) against the oracle, on a grid that fills one tile and leaves a ragged
one, with and without a predictor, by the parity tests' checks (peaks identical but
for near-ties of the FP64 plane, 1e-3 px at agreeing peaks of well-conditioned
windows)."""
import pytest

import oracle
import synth
from test_gpu_parity import check_fp32_pass, compare_pass

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2504_17987_gb300 import build
    build.build()
    oracle.build()
    synth.build()


@pytest.mark.parametrize("radius", [1, 2, 3, 4, 6, 8])
@pytest.mark.parametrize("block", [8, 12, 16, 24, 32])
def test_specialised_shapes_match_the_oracle(block, radius):
    w, s = 2 * block, block
    W, H = 11 * s + 2 * radius + 5, 6 * s + 2 * radius + 9
    W, H = max(W, w + 2 * radius + 4), max(H, w + 2 * radius + 4)
    k = min(1.0, (radius - 0.4) / 3.0)
    flow = synth.Flow(U=1.7 * k, V=-0.9 * k, vortices=[(0.5 * W, 0.5 * H, 20.0 * k, 20.0)])
    A, B = synth.render_pair(synth.ImageSpec(W=W, H=H, bit_depth=8, ppp=0.05, dp=(2.5, 2.5), seed=500 + block + radius), flow)
    nx, ny = oracle.grid_n(W, w, s), oracle.grid_n(H, w, s)
    r = synth.uniform(7, 2 * nx * ny).reshape(2, ny, nx)
    check_fp32_pass(compare_pass(A, B, w, s, radius, None, None), radius)
    pu, pv = 1.7 * k + 0.3 * (r[0] - 0.5), -0.9 * k + 0.3 * (r[1] - 0.5)
    check_fp32_pass(compare_pass(A, B, w, s, radius, pu, pv), radius)
