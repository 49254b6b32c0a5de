"""Encoder: rows that are decided with the IEEE quotient, by the whole warp.  Values on and one step off the midpoints of the code book, in every lane
and place, many in a row; block maxima whose reciprocal is not a normal number in one half of a row or in both."""
import numpy as np
import pytest
import torch

from paper_2311_12023_b200 import binding, inputs
from test_gpu_codec import C
from gpu_util import encode_both

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("b0", [2, 3, 4, 8])
@pytest.mark.parametrize("B0", [16, 32, 64, 256])
@pytest.mark.parametrize("share", [0.002, 0.2, 1.0])
def test_values_at_midpoints(b0, B0, share):
    N, K = 136, 512
    rng = np.random.default_rng(b0 * 1000 + B0)
    cb = binding.nf_codebook(b0)
    mid = ((cb[1:].astype(np.float64) + cb[:-1]) / 2).astype(np.float32)
    A = rng.standard_normal((N, K)).astype(np.float32)
    A /= np.abs(A).reshape(-1, B0).max(axis=1).repeat(B0).reshape(N, K)          # block maxima 1
    at = mid[rng.integers(0, len(mid), (N, K))]
    at = np.where(rng.random((N, K)) < 0.5, at, np.nextafter(at, rng.choice([-2.0, 2.0], (N, K)).astype(np.float32)))
    A = np.where((rng.random((N, K)) < share) & (np.abs(A) < 1), at, A).astype(np.float32)
    A.reshape(-1, B0)[:, 3] = np.where(np.abs(A.reshape(-1, B0)).max(axis=1) < 1, 1.0, A.reshape(-1, B0)[:, 3])
    A *= rng.choice([0.5, 1.0, 2.0], (N, 1)).astype(np.float32)
    encode_both(A, C(b0, B0, 8, 16, 32))


@pytest.mark.parametrize("b0", [2, 3, 4, 8])
@pytest.mark.parametrize("B0", [16, 32, 128])
def test_reciprocals_that_are_not_normal(b0, B0):
    N, K = 64, 256
    rng = np.random.default_rng(7 + b0)
    A = rng.standard_normal((N, K)).astype(np.float32)
    scale = rng.choice(np.array([1.0, 1e-35, 1e-40, 1e32, 0.0], np.float32), N * K // B0).repeat(B0).reshape(N, K)
    encode_both((A * scale).astype(np.float32), C(b0, B0, 8, 64, 32))


# up to eight such rows of a warp are decided by all its lanes together, more by a lane each
@pytest.mark.parametrize("b0", [2, 3, 4, 8])
@pytest.mark.parametrize("rows", [1, 7, 8, 9, 31, 32])
def test_number_of_marked_rows(b0, rows):
    N, K, B0 = 96, 320, 32
    rng = np.random.default_rng(50 * b0 + rows)
    cb = binding.nf_codebook(b0)
    mid = ((cb[1:].astype(np.float64) + cb[:-1]) / 2).astype(np.float32)
    A = rng.standard_normal((N // 32, 32, K // 32, 32)).astype(np.float32)
    A /= np.abs(A).max(axis=3, keepdims=True)
    for i in range(A.shape[0]):
        for k in range(A.shape[2]):
            for row in rng.permutation(32)[:rows]:
                if k % 5 == 0:
                    A[i, row, k] *= np.float32(1e-36)                            # the whole row
                else:
                    j = rng.permutation(32)[:k]
                    A[i, row, k, j] = rng.choice(mid, k)
                    A[i, row, k, (j[0] + 1) % 32] = 1.0
    encode_both(A.reshape(N, K), C(b0, B0, 8, 16, 32))


def test_matrices_that_are_decided_exactly_take_a_few_times_as_long():
    """Measured: 3.9 to 5 times as long; 38 to 85 when a warp hands the codes of all its rows over one by one."""
    def us(W, cfg):
        ws = torch.empty(binding.packed_sizes(*W.shape, cfg)[3], dtype=torch.uint8, device="cuda")
        times = []
        for _ in range(12):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(4):
                binding.encode(W, cfg, workspace=ws)
            b.record()
            b.synchronize()
            times.append(a.elapsed_time(b) * 250)
        return sorted(times)[3]

    W = torch.randn(4096, 4096, generator=torch.Generator(device="cuda").manual_seed(6), device="cuda")
    for b0 in (2, 3, 4, 8):
        cfg = C(b0, 64, 8, 256, 32)
        assert us(W * 1e-36, cfg) < 12 * us(W, cfg)
