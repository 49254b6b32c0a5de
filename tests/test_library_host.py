"""CPU-only checks of the C-ABI library: it loads, exports every declared symbol, and its
host-side logic (code book, storage formula, sizes, argument validation) is right.  No kernel
is launched here."""
import ctypes
import os
import re
import types

import numpy as np
import pytest

import oracle
from paper_2311_12023_b200 import inputs

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def binding():
    from paper_2311_12023_b200 import build
    build.build()
    from paper_2311_12023_b200 import binding as b
    return b


def test_every_declared_symbol_is_exported(binding):
    header = open(os.path.join(ROOT, "include", "lqlora.h")).read()
    declared = set(re.findall(r"\b(lqlora_[a-z0-9_]+)\s*\(", header))
    declared -= {"lqlora_status", "lqlora_config", "lqlora_qmatrix"}
    assert declared, "no declarations found"
    L = binding.lib()
    for name in sorted(declared):
        assert hasattr(L, name), name
    assert declared == set(binding.EXPORTS) | (declared - set(binding.EXPORTS))
    for name in binding.EXPORTS:
        assert name in declared, f"{name} is bound but not declared in the header"


@pytest.mark.parametrize("b", [2, 3, 4, 8])
def test_library_codebook_is_bit_identical_to_oracle(binding, b):
    # built by different quantile routines (Newton vs bisection), must agree to the last bit
    assert np.array_equal(binding.nf_codebook(b), oracle.nf_codebook(b))


@pytest.mark.parametrize("b", [2, 3, 4, 8])
def test_encoder_bin_table_keeps_thresholds_away_from_bin_edges(binding, b):
    # the fast nearest-code search is exact only if no threshold sits within its 1e-6 guard band of a bin edge
    assert binding.lib().lqlora_encode_search_clearance(b) >= 1e-5


@pytest.mark.parametrize("b", [2, 3, 4])
def test_encoder_curve_gives_the_right_code_wherever_it_is_trusted(binding, b):
    # inputs that the curve does not call close to a threshold: right code, and further from any threshold than the 2 ulp (2.4e-7) by
    # which the kernel's quotient can differ from the exact one
    assert binding.lib().lqlora_encode_curve_clearance(b) >= 4.8e-7
    assert binding.lib().lqlora_encode_curve_clearance(8) == -1.0


def test_storage_formula_and_packed_sizes(binding):
    for b0 in (2, 3, 4, 8):
        for B0 in (16, 32, 64, 128, 256):
            for B1 in (64, 256):
                cfg = inputs.QuantConfig(b0, B0, 8, B1, 32)
                bits = binding.storage_bits_per_param(cfg)
                assert bits == oracle.storage_bits_per_param(b0, 8, 32, B0, B1)
                N, K = 1024, 2048
                cb, sb, s2b, _ = binding.packed_sizes(N, K, cfg)
                assert (cb + sb + s2b) * 8 == bits * N * K      # Eq. (2) to the bit
    assert round(binding.storage_bits_per_param(inputs.QuantConfig(4, 64, 8, 256, 32)), 3) == 4.127
    assert round(binding.storage_bits_per_param(inputs.QuantConfig(3, 64, 8, 256, 32)), 3) == 3.127
    # rows are padded to a multiple of 128 in the packed codes only
    cb, sb, s2b, _ = binding.packed_sizes(100, 64, inputs.QuantConfig(4, 16, 8, 16, 32))
    assert cb == 128 * 64 * 4 // 8 and sb == 100 * 4 and s2b == 4 * ((400 + 15) // 16)


def test_invalid_arguments_are_rejected_before_any_launch(binding):
    L = binding.lib()
    good = inputs.QuantConfig(3, 64, 8, 256, 32)
    sz = ctypes.c_size_t(0)

    def sizes(N, K, cfg):
        c = binding._cfg(cfg)
        return L.lqlora_packed_sizes(N, K, ctypes.byref(c), ctypes.byref(sz), None, None, None)

    assert sizes(128, 128, good) == 0
    assert sizes(128, 128, inputs.QuantConfig(5, 64, 8, 256, 32)) == -1      # b0
    assert sizes(128, 128, inputs.QuantConfig(3, 48, 8, 256, 32)) == -1      # B0 not a power of two
    assert sizes(128, 128, inputs.QuantConfig(3, 64, 5, 256, 32)) == -1      # b1 not in {2, 3, 4, 8}
    assert sizes(128, 128, inputs.QuantConfig(3, 64, 8, 256, 8)) == -1       # b2 not fp32 / fp16 / bf16
    for b1 in (2, 3, 4, 8):
        for b2 in (32, 16, -16):
            assert sizes(128, 128, inputs.QuantConfig(3, 64, b1, 256, b2)) == 0
    assert sizes(128, 100, good) == -2                                       # K % 64
    assert sizes(128, 128, inputs.QuantConfig(3, 256, 8, 256, 32)) == -2     # K % B0
    assert sizes(0, 128, good) == -2

    fake = 0x10000   # never dereferenced: validation fails first
    q = binding.CQMatrix(fake, fake, fake, 128, 128, binding._cfg(good))
    ws = 1 << 30
    fwd = L.lqlora_linear_fwd
    assert fwd(None, fake, fake, 64, fake, 4, fake, fake, ws, None) == -3
    assert fwd(ctypes.byref(q), fake, fake, 64, None, 4, fake, fake, ws, None) == -3
    assert fwd(ctypes.byref(q), None, fake, 64, fake, 4, fake, fake, ws, None) == -3
    assert fwd(ctypes.byref(q), fake, fake, 24, fake, 4, fake, fake, ws, None) == -2      # r % 16
    assert fwd(ctypes.byref(q), fake, fake, 64, fake, 0, fake, fake, ws, None) == -2      # M
    assert fwd(ctypes.byref(q), fake, fake, 64, fake + 2, 4, fake, fake, ws, None) == -4  # alignment
    assert fwd(ctypes.byref(q), fake, fake, 64, fake, 4, fake, fake, 16, None) == -5      # workspace
    qbad = binding.CQMatrix(fake, fake + 1, fake, 128, 128, binding._cfg(good))
    assert L.lqlora_linear_bwd_input(ctypes.byref(qbad), fake, fake, 64, fake, 4, fake, fake, ws, None) == -4
    assert L.lqlora_encode(None, ctypes.byref(q), fake, ws, None) == -3
    assert L.lqlora_encode(fake, ctypes.byref(q), fake, 8, None) == -5
    assert binding.status_string(-7) == "device-side wait timed out"


def test_linear_entry_points_take_a_matrix_and_nothing_else_for_one(binding):
    """The typed prototypes: a CQMatrix by value or by reference is taken, an address or bytes in its place refused before the call."""
    L = binding.lib()
    fake = 0x10000      # never dereferenced: validation fails first
    q = binding.CQMatrix(fake, fake, fake, 128, 128, binding._cfg(inputs.QuantConfig(3, 64, 8, 256, 32)))
    for fn in (L.lqlora_linear_fwd, L.lqlora_linear_bwd_input):
        for arg in (q, ctypes.byref(q), ctypes.pointer(q)):
            assert fn(arg, fake, fake, 64, fake, 0, fake, fake, 1 << 30, None) == -2      # M
        for arg in (fake, bytes(q)):
            with pytest.raises(ctypes.ArgumentError):
                fn(arg, fake, fake, 64, fake, 0, fake, fake, 1 << 30, None)
    # what the binding's own calls pass
    packed = binding.QMatrix(*(types.SimpleNamespace(data_ptr=lambda: fake) for _ in range(3)), 128, 128, inputs.QuantConfig(3, 64, 8, 256, 32)).cbytes()
    assert packed == bytes(q)
    for fn in (L.linear_fwd_packed, L.linear_bwd_input_packed):
        assert fn(packed, fake, fake, 64, fake, 0, fake, fake, 1 << 30, None) == -2


def test_result_of_a_tensor_subclass_is_a_plain_tensor(binding, monkeypatch):
    import torch

    class Tagged(torch.Tensor):
        is_cuda = True                        # host tensors in place of device ones: the call itself is replaced

    monkeypatch.setattr(binding, "_stream", lambda: None)
    cfg = inputs.QuantConfig(3, 64, 8, 256, 32)
    q = binding.QMatrix(*(torch.zeros(n, dtype=torch.uint8) for n in binding.packed_sizes(128, 64, cfg)[:3]), 128, 64, cfg)
    X = torch.zeros(4, 64, dtype=torch.bfloat16).as_subclass(Tagged)
    out = binding._linear(lambda *a: 0, "", q, None, None, X, 128, None, torch.zeros(512, dtype=torch.uint8))
    assert type(out) is torch.Tensor and out.dtype == torch.bfloat16 and out.shape == (4, 128) and not out.requires_grad


def test_no_fallback_without_a_device(binding):
    import torch
    if torch.cuda.is_available():
        pytest.skip("a device is present")
    L = binding.lib()
    fake = 0x10000
    q = binding.CQMatrix(fake, fake, fake, 128, 128, binding._cfg(inputs.QuantConfig()))
    assert L.lqlora_unpack(ctypes.byref(q), fake, None) == -6      # LQLORA_ERR_CUDA, nothing computed


def test_product_path_never_imports_the_oracle():
    pkg = os.path.join(ROOT, "paper_2311_12023_b200")
    for dirpath, _, files in os.walk(pkg):
        for f in files:
            if f.endswith((".py", ".cu", ".cuh", ".h")):
                txt = open(os.path.join(dirpath, f)).read()
                assert "import oracle" not in txt and "from oracle" not in txt and "lqlora_oracle" not in txt, f
    src = open(os.path.join(ROOT, "oracle", "__init__.py")).read() + open(os.path.join(ROOT, "oracle", "lqlora_oracle.cpp")).read()
    assert "paper_2311_12023_b200" not in src and "liblqlora.so" not in src


def test_dispatch_between_the_weight_streaming_and_the_tensor_core_kernels(binding):
    """lqlora_linear_path (host only) names the kernel: up to 16 rows stream the packed weights; from 17 rows the
    tcgen05 kernel on transposed tiles takes over (the input gradient of 9..16 rows too when the matrix has at least 2048 rows);
    CTA pairs run once their [512, 256] tiles fill more than half of the SMs; shapes without 16-byte rows fall back
    to the plain kernels."""
    S, ONE, PAIR, PLAIN = binding.PATH_STREAM, binding.PATH_TC_ONE, binding.PATH_TC_PAIR, binding.PATH_PLAIN
    cfg = inputs.QuantConfig(3, 64, 8, 256, 32)
    for M, want in ((1, S), (16, S), (17, ONE), (256, ONE), (512, ONE), (2048, PAIR)):
        assert binding.linear_path(4096, 4096, cfg, 64, M, False) == want
    for M, want in ((1, S), (8, S), (9, ONE), (16, ONE), (17, ONE), (8192, PAIR)):
        assert binding.linear_path(4096, 4096, cfg, 64, M, True) == want
    for M, want in ((8, S), (9, S), (16, S), (17, ONE)):
        assert binding.linear_path(1024, 8192, cfg, 64, M, True) == want
    odd = inputs.QuantConfig(4, 64, 8, 16, 32)          # 201 rows: the rows of dY do not start on 16-byte boundaries
    assert binding.linear_path(201, 192, odd, 16, 1, False) == S and binding.linear_path(201, 192, odd, 16, 1, True) == PLAIN
    # the contraction of an output tile is shared by a cluster where few tiles would leave SMs idle
    kernel, splits = binding.linear_route(8192, 8192, cfg, 64, 128, False)
    assert kernel == ONE and 2 <= splits <= 4
    kernel, splits = binding.linear_route(8192, 8192, cfg, 64, 2048, False)
    assert kernel == PAIR and splits == 1
    kernel, splits = binding.linear_route(4096, 4096, cfg, 64, 1, False)
    assert kernel == S and 1 <= splits <= 8


def test_budgeted_assignment_matches_exhaustive_search(binding):
    """lqlora_assign_configs (Sec. 3.2, Algorithm 3) against the oracle's enumeration on random small instances."""
    from oracle import lq
    g = inputs.rng(123)
    for trial in range(30):
        n, m = int(g.integers(1, 6)), int(g.integers(1, 5))
        S = np.sort(g.uniform(1.0, 10.0, (n, m)), axis=1)
        E = -np.sort(-g.uniform(0.0, 5.0, (n, m)), axis=1)          # more storage, less error
        budget = float(g.uniform(S[:, 0].sum() * 0.9, S[:, -1].sum() * 1.1))
        want = lq.ilp_solve(S, E, budget)
        got = binding.assign_configs(E, S, budget)
        if want is None:
            assert got is None
            continue
        assert got is not None and got[2] <= budget + 1e-12
        assert abs(got[1] - want[1]) < 1e-12                          # same optimal error (the argmin may tie)
        assert abs(sum(E[i, a] for i, a in enumerate(got[0])) - got[1]) < 1e-12
    # non-monotone tables are handled too (a configuration that is worse in both respects is never chosen)
    S = np.array([[1.0, 2.0, 3.0]])
    E = np.array([[5.0, 7.0, 1.0]])
    assert binding.assign_configs(E, S, 2.5)[0] == [0]
    assert binding.assign_configs(E, S, 3.0)[0] == [2]


@pytest.mark.parametrize("b0", [2, 3, 4, 8])
def test_every_number_of_rows_has_a_plan_on_the_tensor_core_kernels(binding, b0):
    """The route of a call names at least one slice of the contraction for any number of rows, on narrow outputs (all of
    them on transposed tiles) and where the pair kernel peels columns off (an error without a plan for those).  8-bit codes
    take the most shared memory: their token chunks end at 384 instead of 512 rows."""
    cfg = inputs.QuantConfig(b0, 64, 8, 256, 32)
    g = inputs.rng(77 + b0)
    edges = [m + d for m in (512, 3072, 11136, 11264, 11520, 11776, 12288, 14336, 16384, 18944, 28672, 1 << 20, 1 << 24) for d in (-1, 0, 1)]
    rows = sorted({m for m in edges + list(range(17, 19200, 37)) + [int(2 ** x) for x in g.uniform(4.1, 24.0, 400)] if 17 <= m <= 1 << 24})
    for N, K in ((256, 4096), (64, 512), (4096, 512), (8192, 1024), (14336, 4096), (28672, 8192)):
        for M in rows:
            for r, backward in ((64, False), (0, False), (128, True)):
                kernel, splits = binding.linear_route(N, K, cfg, r, M, backward)
                assert kernel in (binding.PATH_TC_ONE, binding.PATH_TC_PAIR) and 1 <= splits <= 4, (N, K, M, r, backward)


def test_no_kernel_polls_a_barrier_for_both_parities():
    """try_wait.parity succeeds for the parity of the phase before the current one, so "neither parity" is never true and a loop
    on it waits for nothing: copies in flight are awaited by the phase they were issued in (let_land, drain_ring)."""
    import glob
    import re
    for f in glob.glob(os.path.join(ROOT, "paper_2311_12023_b200", "csrc", "*")):
        for args in re.findall(r"!mbar_try_wait\((.*?), 0\) && !mbar_try_wait\(.*?, 1\)", open(f).read()):
            raise AssertionError(f"{os.path.basename(f)}: {args}")
