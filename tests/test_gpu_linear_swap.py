"""tcgen05 kernel on transposed output tiles: tile edges, token boxes, slices of the contraction, rank-r steps."""
import pytest

from paper_2311_12023_b200 import binding, inputs
from test_gpu_linear import C, run_case

pytestmark = pytest.mark.gpu


# rows on both sides of a box (16), of one / two boxes (256 / 257) and of one / two chunks (512 / 513); an odd number of
# 128-column tiles (the second CTA of the last pair has none) and a last tile of 64 columns
@pytest.mark.parametrize("N,K,M", [(384, 448, 17), (392, 1984, 33), (136, 4096, 256), (136, 4096, 257), (640, 320, 512), (328, 704, 513)])
@pytest.mark.parametrize("b0,B0", [(3, 64), (4, 16), (2, 32), (8, 64)])
def test_tile_box_and_slice_edges(N, K, M, b0, B0):
    cfg = C(b0, B0, 8, 64, 32)
    assert binding.linear_path(N, K, cfg, 64, M, False) == binding.PATH_TC_ONE
    assert binding.linear_path(N, K, cfg, 64, M, True) == binding.PATH_TC_ONE
    A = inputs.gaussian(1600 + N, (N, K), 0.02)
    l1b, l2b = inputs.lowrank_factors(1601 + K, N, K, 64, 0.01)
    run_case(A, l1b, l2b, cfg, M, seed=1700 + M)


# ranks that fill a part of one 64-wide step, exactly one, and two; and none
@pytest.mark.parametrize("r", [0, 16, 64, 80, 128])
def test_rank_steps(r):
    N, K, M = 520, 1088, 100
    A = inputs.student_t(1650, (N, K), 5.0, 0.02)
    l1b, l2b = inputs.lowrank_factors(1651, N, K, r, 0.03) if r else (None, None)
    run_case(A, l1b, l2b, C(3, 64, 8, 256, 32), M, seed=1750 + r)


# 8-bit codes take the most shared memory (token chunks of at most 384 rows): many rows on a narrow output, and on the columns
# that the pair kernel peels off (4096 columns at 12288 rows: 384 pair tiles, 14 of them in the last wave), both passes
@pytest.mark.parametrize("N,K", [(256, 512), (512, 256), (4096, 512), (512, 4096)])
def test_8_bit_codes_many_rows(N, K):
    M = 12288
    A = inputs.gaussian(1800 + N, (N, K), 0.02)
    l1b, l2b = inputs.lowrank_factors(1801 + K, N, K, 64, 0.01)
    route = {256: binding.PATH_TC_ONE, 4096: binding.PATH_TC_PAIR}.get(N)
    run_case(A, l1b, l2b, C(8, 64, 8, 64, 32), M, seed=1810, rows=inputs.sample_rows(1811, M, count=24, tile=384), route=route)
