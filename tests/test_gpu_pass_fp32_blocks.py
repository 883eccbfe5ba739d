"""The FP32 pass kernels that are not specialised to one shape, against the oracle by the
parity tests' checks: blocks of 8, 12, 16 and 24 px at other overlaps than 50 % (the
kernel with the unrolled loops) and blocks of 4, 20, 28 and 32 px (the other one), on
grids of tiles with and without 16 windows."""
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


SHAPES = [(32, 8, 1), (32, 8, 4), (24, 8, 6), (48, 12, 2), (48, 12, 8), (16, 16, 3), (64, 16, 4), (96, 24, 6),  # unrolled
          (16, 4, 0), (16, 4, 1), (16, 4, 4), (24, 4, 3), (12, 4, 2), (12, 4, 8), (40, 20, 3), (20, 20, 4), (56, 28, 6), (32, 32, 4)]


def case(w, s, radius):
    W, H = w + max(18 * s, 2 * radius + 4) + 5, w + max(9 * s, 2 * radius + 4) + 3
    flow = synth.Flow(U=1.4, V=-0.8)
    A, B = synth.render_pair(synth.ImageSpec(W=W, H=H, bit_depth=8, ppp=0.12, dp=(2.5, 2.5), seed=700 + 40 * w + s + radius), flow)
    nx, ny = oracle.grid_n(W, w, s), oracle.grid_n(H, w, s)
    r = synth.uniform(w + s + radius, 2 * nx * ny).reshape(2, ny, nx)
    return A, B, 1.4 + 0.3 * (r[0] - 0.5), -0.8 + 0.3 * (r[1] - 0.5)


@pytest.mark.parametrize("w, s, radius", SHAPES)
def test_block_sizes_match_the_oracle(w, s, radius):
    A, B, pu, pv = case(w, s, radius)
    check_fp32_pass(compare_pass(A, B, w, s, radius, pu, pv), radius)
