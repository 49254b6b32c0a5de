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
