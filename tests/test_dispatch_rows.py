"""The line between transposed tiles and CTA pairs (estimated times below 2048 rows): routes, and results on both sides of it."""
import pytest

from paper_2311_12023_b200 import binding, inputs
from test_gpu_linear import C, run_case

ONE, PAIR = binding.PATH_TC_ONE, binding.PATH_TC_PAIR


@pytest.mark.parametrize("N,K,b0,M,want", [
    (8192, 8192, 3, 520, ONE), (8192, 8192, 3, 1024, PAIR), (8192, 8192, 3, 1100, ONE), (8192, 8192, 3, 1400, ONE),       # one wave of pairs / the second
    (8192, 8192, 3, 2048, PAIR), (8192, 8192, 8, 1100, ONE), (5120, 5120, 2, 700, ONE), (5120, 5120, 2, 1400, PAIR),
    (28672, 8192, 3, 2047, PAIR), (256, 4096, 3, 4096, ONE)])                                                             # few tiles: always transposed
def test_route_between_256_and_2048_rows(N, K, b0, M, want):
    assert binding.linear_path(N, K, C(b0, 64, 8, 256, 32), 64, M, False) == want


# from 2048 rows on the pairs, also where their last wave is between a quarter and a half full
@pytest.mark.parametrize("N,K,b0,M", [(4392, 26688, 8, 2579), (2040, 27008, 3, 2251), (8192, 28672, 8, 2300), (5120, 5120, 8, 2100), (4096, 11008, 8, 2600)])
def test_pairs_from_2048_rows(N, K, b0, M):
    assert binding.linear_path(N, K, C(b0, 64, 8, 256, 32), 64, M, False) == PAIR


# few rows against a long contraction: sliced over clusters although these need a second wave
@pytest.mark.parametrize("N,K,b0,B0,M,r,backward", [(9472, 16640, 3, 16, 30, 0, False), (9088, 16896, 2, 64, 19, 64, False), (8264, 10752, 3, 256, 17, 64, False),
                                                    (8320, 22272, 8, 64, 24, 64, True)])
def test_long_contractions_of_few_rows_are_sliced(N, K, b0, B0, M, r, backward):
    kernel, splits = binding.linear_route(N, K, C(b0, B0, 8, 256, 32), r, M, backward)
    assert kernel == ONE and splits > 1


# calls where another kernel or another number of slices, taken by an earlier model of the split, cost 10 to 47 %
@pytest.mark.parametrize("N,K,b0,B0,M,r,backward,want", [
    (13848, 4224, 4, 128, 601, 64, False, (ONE, 1)), (4784, 21120, 8, 64, 445, 64, False, (ONE, 3)), (13240, 11968, 2, 64, 773, 16, False, (ONE, 1)),
    (22904, 10048, 8, 32, 301, 64, False, (ONE, 2)), (2688, 2304, 2, 32, 283, 64, False, (ONE, 2)), (9216, 16896, 4, 32, 19, 16, True, (ONE, 1)),
    (3456, 1792, 8, 64, 808, 128, True, (ONE, 2)), (16648, 8768, 8, 32, 628, 64, True, (ONE, 1)), (14336, 15616, 4, 128, 884, 64, True, (ONE, 1)),
    (16512, 1792, 2, 64, 32, 0, False, (ONE, 1))])
def test_slices_of_the_contraction(N, K, b0, B0, M, r, backward, want):
    assert binding.linear_route(N, K, C(b0, B0, 8, 256, 32), r, M, backward) == want


# many chunks of transposed tiles where the pairs ran before: a last chunk that is not full, both passes, rank below and above 64
@pytest.mark.gpu
@pytest.mark.parametrize("N,K,b0,M,r", [(8192, 2048, 3, 1100, 64), (5120, 1024, 2, 700, 128), (8200, 1024, 8, 1101, 16)])
def test_transposed_tiles_in_place_of_pairs(N, K, b0, M, r):
    cfg = C(b0, 64, 8, 64, 32)
    assert binding.linear_path(N, K, cfg, r, M, False) == ONE
    A = inputs.gaussian(7100 + N, (N, K), 0.02)
    l1b, l2b = inputs.lowrank_factors(7101, N, K, r, 0.03) if r else (None, None)
    run_case(A, l1b, l2b, cfg, M, seed=7200, rows=inputs.sample_rows(7201, M, count=24, tile=128))
