"""The 16-bit pass kernels that are not specialised to one block size, against the
oracle by the parity tests' checks: from r = 4 on, blocks whose fragments come by
ldmatrix (multiples of 16 px; 8 px up to r = 6) and the others have kernels of their own;
window sizes with and without the unrolled stencil in each."""
import pytest

import oracle
import synth
from test_gpu_parity import check_16bit_pass, compare_pass

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2504_17987_gb300 import build
    build.build()
    oracle.build()
    synth.build()


SHAPES = [(32, 8, 4), (64, 16, 4), (48, 48, 4), (24, 8, 6), (16, 8, 6), (32, 16, 6), (64, 32, 6), (96, 48, 6), (32, 16, 8), (64, 16, 8),  # ldmatrix
          (24, 12, 4), (24, 6, 4), (16, 4, 4), (28, 14, 4), (24, 12, 6), (20, 10, 6), (16, 8, 8), (32, 8, 8), (48, 24, 8), (36, 18, 8)]  # the rest


def case(w, s, radius):
    W, H = w + max(12 * s, 2 * radius + 4) + 5, w + max(10 * s, 2 * radius + 4) + 3
    flow = synth.Flow(U=1.4, V=-0.8)
    A, B = synth.render_pair(synth.ImageSpec(W=W, H=H, bit_depth=8, ppp=0.12, dp=(2.5, 2.5), seed=900 + 40 * w + s + radius), flow)
    nx, ny = oracle.grid_n(W, w, s), oracle.grid_n(H, w, s)
    r = synth.uniform(w + s + radius, 2 * nx * ny).reshape(2, ny, nx)
    return A, B, 1.4 + 0.3 * (r[0] - 0.5), -0.8 + 0.3 * (r[1] - 0.5)


@pytest.mark.parametrize("w, s, radius", SHAPES)
def test_block_sizes_match_the_oracle(w, s, radius):
    A, B, pu, pv = case(w, s, radius)
    check_16bit_pass(compare_pass(A, B, w, s, radius, pu, pv, precision="bf16"), radius, "bf16")
