"""Encoder at the decision thresholds: inputs on both sides of every midpoint of the code book, where the fast search has to hand over to
the IEEE quotient."""
import numpy as np
import pytest

from paper_2311_12023_b200 import binding, inputs
from gpu_util import encode_both

pytestmark = pytest.mark.gpu


# block maxima: powers of two (exact reciprocals), others, and two whose reciprocal is not a normal number
@pytest.mark.parametrize("b0,B0", [(2, 16), (2, 64), (3, 16), (3, 32), (3, 256), (4, 16), (4, 64), (8, 64)])
def test_codes_next_to_the_thresholds(b0, B0):
    cb = binding.nf_codebook(b0).astype(np.float64)
    mid = (cb[1:] + cb[:-1]) / 2
    steps = np.concatenate([np.arange(-12, 13), 2 ** np.arange(4, 12), -2 ** np.arange(4, 12)])
    N, K = 160, 256
    g = inputs.rng(4100 + b0)
    A = np.zeros((N * K // B0, B0), dtype=np.float32)
    for i in range(A.shape[0]):
        s = np.float32([1.0, 0.25, 0.0371, 1.7e-3, 3.3e4, 1e-33, 1e-39][i % 7] * (1.0 if i % 7 < 2 else g.uniform(0.5, 1.0)))
        t = np.float32(mid[g.integers(0, len(mid), B0)] * np.float64(s))
        ulp = np.spacing(np.abs(t))
        A[i] = t + np.float32(g.choice(steps, B0)) * ulp
        A[i] = np.clip(A[i], -s, s)
        A[i, g.integers(0, B0)] = s if i % 2 else -s
    encode_both(A.reshape(N, K), inputs.QuantConfig(b0, B0, 8, 64, 32))
