"""FP32 passes whose blocks are not a multiple of 4 px (the kernel of any radius)
against the oracle, on grids of several tiles of 16 and more windows, by the parity
tests' checks (peaks identical but for near-ties of the FP64 plane, 1e-3 px at agreeing
peaks of well-conditioned windows)."""
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


def case(w, s, radius):
    W, H = w + 18 * s + 5, w + 12 * s + 3
    flow = synth.Flow(U=1.4, V=-0.8)
    A, B = synth.render_pair(synth.ImageSpec(W=W, H=H, bit_depth=8, ppp=0.12, dp=(2.5, 2.5), seed=40 * w + radius), flow)
    nx, ny = oracle.grid_n(W, w, s), oracle.grid_n(H, w, s)
    r = synth.uniform(w + radius, 2 * nx * ny).reshape(2, ny, nx)
    return A, B, 1.4 + 0.3 * (r[0] - 0.5), -0.8 + 0.3 * (r[1] - 0.5)


SHAPES = [(20, 10, 4), (12, 6, 2), (14, 7, 3), (18, 9, 1), (22, 11, 4), (20, 5, 1), (20, 5, 0), (28, 7, 1), (20, 10, 3)]


@pytest.mark.parametrize("w, s, radius", SHAPES)
def test_blocks_off_a_multiple_of_four_match_the_oracle(w, s, radius):
    A, B, pu, pv = case(w, s, radius)
    check_fp32_pass(compare_pass(A, B, w, s, radius, pu, pv), radius)
