"""Weight-streaming kernels: edges of units, runs, scale runs, second-level groups and rank-r units."""
import numpy as np
import pytest
import torch

from paper_2311_12023_b200 import binding, inputs
from test_gpu_linear import C, run_case

pytestmark = pytest.mark.gpu


# one tile of a unit / of a window, a ragged last unit, a partial tile row and slab; rows of blocks that are not whole vectors of scale
# codes (odd numbers of blocks, groups of 16 blocks that end inside a vector); tokens on both sides of 8; fewer units than SMs, one tile
# row shared by all runs (40960 columns), runs over three tile rows (40000 rows)
@pytest.mark.parametrize("N,K,M", [(8, 64, 1), (40, 192, 8), (136, 1088, 7), (392, 1984, 9), (1000, 320, 16), (264, 2368, 3),
                                   (64, 40960, 2), (40000, 64, 5)])
@pytest.mark.parametrize("b0,B0,B1,r", [(2, 16, 64, 16), (2, 64, 16, 80), (3, 64, 16, 64), (3, 32, 256, 128), (4, 16, 16, 48), (4, 64, 64, 0), (8, 64, 16, 16)])
def test_unit_run_and_scale_edges(N, K, M, b0, B0, B1, r):
    cfg = C(b0, B0, 8, B1, 32)
    assert binding.linear_path(N, K, cfg, r, M, False) == binding.PATH_STREAM
    A = inputs.gaussian(6100 + N, (N, K), 0.02)
    l1b, l2b = inputs.lowrank_factors(6101 + K, N, K, r, 0.05) if r else (None, None)
    run_case(A, l1b, l2b, cfg, M, seed=6200 + M)


# blocks wider than a tile and than a window, on a matrix whose runs end inside a tile row, both sides of eight tokens
@pytest.mark.parametrize("M", [1, 8, 9, 16])
@pytest.mark.parametrize("b0,B0", [(2, 128), (3, 256), (4, 128), (8, 256)])
def test_wide_blocks(b0, B0, M):
    N, K = 1928, 2304
    A = inputs.student_t(6300 + b0, (N, K), 5.0, 0.02)
    l1b, l2b = inputs.lowrank_factors(6301, N, K, 64, 0.03)
    run_case(A, l1b, l2b, C(b0, B0, 8, 16, 32), M, seed=6400 + M)


# more units than the SMs can take in one run each (two and more runs per CTA, with buffers used again), and tiles that are given to a run
# whole because the slots would exceed their room (one slot), in both directions, with and without a rank-r term
@pytest.mark.parametrize("N,K,M,backward,whole", [(60000, 320, 1, False, False), (60000, 320, 5, False, False), (60000, 320, 16, False, True),
                                                  (64, 53248, 8, True, False), (64, 53248, 16, True, True)])
@pytest.mark.parametrize("r", [0, 32])
def test_several_runs_per_cta_and_whole_tiles(N, K, M, backward, whole, r):
    cfg = C(3, 64, 8, 64, 32)
    kernel, slots = binding.linear_route(N, K, cfg, r, M, backward)
    assert kernel == binding.PATH_STREAM and (slots == 1) == whole
    A = inputs.gaussian(6560 + M, (N, K), 0.02)
    l1b, l2b = inputs.lowrank_factors(6561, N, K, r, 0.05) if r else (None, None)
    run_case(A, l1b, l2b, cfg, M, seed=6562, passes=("bwd",) if backward else ("fwd",))


# sixteen rows of a long contraction: a run has more units than there is room for activations, which are staged in turns
@pytest.mark.parametrize("b0", [3, 8])
def test_activations_staged_in_turns(b0):
    N, K, M = 3200, 28672, 16
    A = inputs.gaussian(6570, (N, K), 0.02)
    l1b, l2b = inputs.lowrank_factors(6571, N, K, 64, 0.02)
    run_case(A, l1b, l2b, C(b0, 64, 8, 256, 32), M, seed=6572, passes=("fwd",), route=binding.PATH_STREAM)


# 8-bit codes: the code book is laid out by CTAs of 8 warps (192 rows: one unit per run; input gradient: up to eight), 12 and 16
@pytest.mark.parametrize("N", [192, 2600, 4096])
def test_code_book_of_eight_bit_codes(N):
    K = 2304
    A = inputs.gaussian(6550, (N, K), 0.02)
    l1b, l2b = inputs.lowrank_factors(6551, N, K, 16, 0.03)
    run_case(A, l1b, l2b, C(8, 64, 8, 64, 32), 3, seed=6552)


# rows of the identity: the weights of the streaming kernels are the bits of lqlora_dequant, which forms the second-level scale v / levels by a
# division.  Many groups, because one unit in the last place of a scale shows in few of the rounded products
@pytest.mark.parametrize("b1", [8, 4])
@pytest.mark.parametrize("b0,B0", [(2, 16), (3, 64), (4, 32), (8, 64)])
def test_identity_rows_return_the_dequantized_weights(b0, B0, b1):
    cfg = C(b0, B0, b1, 16, 32)
    for N, K, backward in ((40000, 64, False), (64, 16384, True)):
        A = inputs.student_t(6590 + b0, (N, K), 5.0, 0.02)
        q = binding.encode(torch.from_numpy(A).cuda(), cfg)
        d16 = binding.dequant(q)[1]
        at = torch.arange(3, 3 + 4 * 16, 4, device="cuda")
        x = torch.zeros(16, N if backward else K, dtype=torch.bfloat16, device="cuda")
        x[torch.arange(16, device="cuda"), at] = 1.0
        assert binding.linear_path(N, K, cfg, 0, 16, backward) == binding.PATH_STREAM
        if backward:
            got, want = binding.linear_bwd_input(q, None, None, x), d16[at]
        else:
            got, want = binding.linear_fwd(q, None, None, x), d16[:, at].T
        assert torch.equal(got, want)


# one tile row / a few windows shared by many runs: slots on both sides of the eight that are summed at a time, last columns of a tile
@pytest.mark.parametrize("M", [1, 5, 16])
@pytest.mark.parametrize("slots", [2, 7, 8, 9, 17])
def test_slots_of_a_shared_tile(slots, M):
    N, K, r = 120, 256 * slots, 32
    cfg = C(3, 64, 8, 64, 32)
    assert binding.linear_route(N, K, cfg, r, M, False) == (binding.PATH_STREAM, slots)
    A = inputs.gaussian(6600 + slots, (N, K), 0.02)
    l1b, l2b = inputs.lowrank_factors(6601, N, K, r, 0.05)
    run_case(A, l1b, l2b, cfg, M, seed=6700 + M, passes=("fwd",))
    # input gradient of the transposed shape: 32 rows per unit, one of them the rank-r term
    N, K = 32 * (slots - 1), 128
    assert binding.linear_route(N, K, cfg, r, M, True) == (binding.PATH_STREAM, slots)
    A = inputs.gaussian(6602 + slots, (N, K), 0.02)
    l1b, l2b = inputs.lowrank_factors(6603, N, K, r, 0.05)
    run_case(A, l1b, l2b, cfg, M, seed=6800 + M, passes=("bwd",))


# block maxima above 65504 with fp16 second-level scales: the group's scale is infinite in lqlora_dequant, and so are its weights;
# the last unit of 320 columns has blocks behind the last one, which must add nothing
@pytest.mark.parametrize("K", [512, 320])
@pytest.mark.parametrize("b0,B0,M", [(2, 16, 1), (2, 64, 16), (3, 64, 3), (4, 32, 1), (8, 64, 9)])
def test_infinite_second_level_scale(b0, B0, M, K):
    N = 256
    cfg = C(b0, B0, 8, 64, 16)
    A = inputs.gaussian(6500, (N, K), 0.02)
    whole = 64 * B0 * K // np.gcd(64 * B0, K) // K               # rows that end where a group ends
    A[:whole] = 7e4
    q = binding.encode(torch.from_numpy(A).cuda(), cfg)
    d16 = binding.dequant(q)[1]
    assert bool(torch.isposinf(d16[:whole]).all()) and bool(torch.isfinite(d16[whole:]).all())
    assert binding.linear_path(N, K, cfg, 0, M, False) == binding.PATH_STREAM
    x = torch.ones(M, K, dtype=torch.bfloat16, device="cuda")
    Y = binding.linear_fwd(q, None, None, x)
    assert bool(torch.isposinf(Y[:, :whole]).all())
    want = x.float() @ d16[whole:].float().T
    assert float((Y[:, whole:].float() - want).norm() / want.norm()) < 5e-3
    dY = torch.ones(M, N, dtype=torch.bfloat16, device="cuda")
    assert bool(torch.isposinf(binding.linear_bwd_input(q, None, None, dY)).all())
