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


# many chunks of transposed tiles where the pairs ran before: a last chunk that is not full, both passes, rank below and above 64
@pytest.mark.gpu
@pytest.mark.parametrize("N,K,b0,M,r", [(8192, 2048, 3, 1100, 64), (5120, 1024, 2, 700, 128), (8200, 1024, 8, 1101, 16)])
def test_transposed_tiles_in_place_of_pairs(N, K, b0, M, r):
    cfg = C(b0, 64, 8, 64, 32)
    assert binding.linear_path(N, K, cfg, r, M, False) == ONE
    A = inputs.gaussian(7100 + N, (N, K), 0.02)
    l1b, l2b = inputs.lowrank_factors(7101, N, K, r, 0.03) if r else (None, None)
    run_case(A, l1b, l2b, cfg, M, seed=7200, rows=inputs.sample_rows(7201, M, count=24, tile=128))
