"""Transposed tiles with the weights in tensor memory (forward, one token box): ring of eight stages, code widths, rank-r steps."""
import pytest

from paper_2311_12023_b200 import binding, inputs
from test_gpu_linear import C, run_case

pytestmark = pytest.mark.gpu


# rows at both ends of a token box (17 .. 256) and just past it (257: two boxes, weights in shared memory); contractions of fewer steps
# than the ring has stages (7), as many (8), one more (9), and sliced ones; last tiles of 8 columns, and pairs whose second CTA has
# none; ranks that end inside the first and inside the second 64-wide step, that fill both, and none
@pytest.mark.parametrize("N,K,M,r", [(392, 448, 17, 16), (640, 512, 31, 80), (136, 576, 255, 128), (264, 4096, 256, 80), (136, 4096, 257, 16),
                                     (2056, 1984, 64, 0)])
@pytest.mark.parametrize("b0,B0", [(2, 64), (3, 16), (4, 32), (8, 16)])
def test_one_token_box(N, K, M, r, b0, B0):
    cfg = C(b0, B0, 8, 64, 32)
    A = inputs.gaussian(2600 + N, (N, K), 0.02)
    l1b, l2b = inputs.lowrank_factors(2601 + K, N, K, r, 0.03) if r else (None, None)
    run_case(A, l1b, l2b, cfg, M, seed=2700 + M, route=binding.PATH_TC_ONE)
