"""Transposed tiles with two steps of 64 contraction elements per stage: odd numbers of steps, rank-r steps that share a stage with the last
weights, calls without a rank-r term one after the other, and scale windows of 16 codes that start and end inside a row."""
import pytest
import torch

from paper_2311_12023_b200 import binding, inputs
from test_gpu_linear import C, run_case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,K,B0", [(136, 192, 64), (264, 320, 16), (200, 1088, 64), (520, 2112, 32), (72, 768, 256), (1160, 1216, 64)])
@pytest.mark.parametrize("b0,M,r", [(3, 17, 0), (2, 40, 16), (4, 100, 80), (8, 33, 128), (3, 250, 64)])
def test_two_steps_per_stage(N, K, B0, b0, M, r):
    cfg = C(b0, B0, 8, 16, 32)
    assert binding.linear_path(N, K, cfg, r, M, False) == binding.PATH_TC_ONE
    A = inputs.gaussian(8100 + N + b0, (N, K), 0.02)
    l1b, l2b = inputs.lowrank_factors(8101 + K, N, K, r, 0.03) if r else (None, None)
    run_case(A, l1b, l2b, cfg, M, seed=8200 + M)


def test_calls_without_rank_term_follow_each_other():
    """Such a call is one kernel, launched while the one in front ends: each reads what the one in front has written."""
    cfg = C(3, 64, 8, 64, 32)
    g = torch.Generator(device="cuda").manual_seed(5)
    qs = [binding.encode(torch.randn(1024, 1024, generator=g, device="cuda") * 0.03, cfg) for _ in range(4)]
    ws = [binding.alloc_workspace(q, 0, 48) for q in qs]
    X = torch.randn(48, 1024, generator=g, device="cuda").to(torch.bfloat16)

    def chain(wait):
        x = X
        for i in range(12):
            x = (binding.linear_fwd if i % 3 else binding.linear_bwd_input)(qs[i % 4], None, None, x, workspace=ws[i % 4])
            if wait:
                torch.cuda.synchronize()
        torch.cuda.synchronize()
        return x

    want = chain(True)
    for _ in range(5):
        assert torch.equal(chain(False), want)
    assert all(binding.workspace_status(w) == 0 for w in ws)


# input gradient: two steps per stage up to 64 tokens of 2-bit codes, one otherwise; one token box and two
@pytest.mark.parametrize("b0,M", [(2, 17), (2, 64), (2, 65), (2, 257), (3, 64), (4, 129), (8, 24), (8, 200), (8, 256), (8, 300)])
@pytest.mark.parametrize("N,K,B0", [(2056, 192, 16), (712, 576, 64)])
def test_steps_per_stage_of_the_input_gradient(N, K, B0, b0, M):
    cfg = C(b0, B0, 8, 64, 32)
    assert binding.linear_path(N, K, cfg, 48, M, True) == binding.PATH_TC_ONE
    A = inputs.gaussian(8300 + N + b0, (N, K), 0.02)
    l1b, l2b = inputs.lowrank_factors(8301 + K, N, K, 48, 0.03)
    run_case(A, l1b, l2b, cfg, M, seed=8400 + M)


def test_more_than_37_row_tiles_of_the_pre_product():
    """One split of the contraction per row tile, whatever the linear kernel leaves idle; the last tile is one row."""
    N, K, M = 512, 512, 4865
    cfg = C(3, 64, 8, 64, 32)
    assert binding.linear_path(N, K, cfg, 64, M, False) == binding.PATH_TC_ONE
    A = inputs.gaussian(8500, (N, K), 0.03)
    l1b, l2b = inputs.lowrank_factors(8501, N, K, 64, 0.03)
    run_case(A, l1b, l2b, cfg, M, seed=8502, rows=inputs.sample_rows(8503, M, count=24, tile=128))
