"""Encoder: rows that are decided with the IEEE quotient, by the whole warp.  Values on and one step off the midpoints of the code book, in every lane
and place, many in a row; block maxima whose reciprocal is not a normal number in one half of a row or in both."""
import numpy as np
import pytest

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
