"""Calls enqueued one behind the other without a synchronisation: the first kernel of a call starts while the last one of the call
before it ends, so each has to wait before it reads what that one writes (the result, the workspace) or overwrites it."""
import types

import numpy as np
import pytest
import torch

from paper_2311_12023_b200 import binding, inputs
from test_gpu_linear import C

pytestmark = pytest.mark.gpu

M, R = 2100, 64


class Layer:
    def __init__(self, seed, N, K, cfg, r=R):
        self.q = binding.encode(torch.from_numpy(inputs.gaussian(seed, (N, K), 0.04)).cuda(), cfg)
        self.r = r
        self.L1 = self.L2 = None
        if r:
            l1b, l2b = inputs.lowrank_factors(seed + 1, N, K, r, 0.02)
            self.L1, self.L2 = binding.bf16_from_bits(l1b), binding.bf16_from_bits(l2b)

    def path(self, rows, backward):
        return binding.linear_path(self.q.N, self.q.K, self.q.cfg, self.r, rows, backward)


class Chain:
    """The calls of one run, in order; every result goes into a buffer that a later call reads."""

    def __init__(self):
        wide, narrow = Layer(9000, 2560, 512, C(3, 64, 8, 256, 32)), Layer(9010, 512, 2560, C(4, 32, 8, 64, 32))
        square, plain = Layer(9020, 512, 512, C(2, 64, 8, 64, 32)), Layer(9030, 512, 512, C(8, 64, 8, 64, 32), r=0)
        packed = Layer(9040, 512, 512, C(3, 64, 4, 64, 16))
        nf8 = C(8, 64, 8, 256, 32)
        f1, f2 = (binding.encode(x.float().contiguous(), nf8) for x in (square.L1, square.L2))
        S, ONE, PAIR = binding.PATH_STREAM, binding.PATH_TC_ONE, binding.PATH_TC_PAIR
        assert wide.path(M, False) == PAIR and narrow.path(M, False) == ONE and square.path(8, False) == S
        assert square.path(100, True) == ONE and narrow.path(M, True) == PAIR and wide.path(M, True) == ONE

        def bf(rows, cols):
            return torch.empty(rows, cols, dtype=torch.bfloat16, device="cuda")

        self.src = binding.bf16_from_bits(inputs.activations(9100, M, 512))
        X, Y1, Y2, Y3, dY1, dX1 = bf(M, 512), bf(M, 2560), bf(M, 512), bf(M, 512), bf(M, 2560), bf(M, 512)
        s = [bf(100, 512) for _ in range(10)]
        g = [torch.empty(*shape, dtype=torch.float32, device="cuda") for shape in ((2560, R), (R, 512), (512, R), (R, 2560))]
        need = max(binding.linear_workspace_bytes(l.q.N, l.q.K, l.q.cfg, l.r, rows) for l in (wide, narrow, square, plain, packed)
                   for rows in (8, 100, M))
        need = max(need, binding.lora_grads_workspace_bytes(2560, 512, R, M))
        ws = torch.empty(need, dtype=torch.uint8, device="cuda")               # one workspace for every call
        ws_f, ws_b = torch.empty_like(ws), torch.empty_like(ws)                # ... but for the two whose intermediates are used
        self.X = X
        self.poisoned = [Y1, Y2, Y3, dY1, dX1] + s + g
        self.results = self.poisoned

        def fwd(l, x, out, w=ws):
            return lambda: binding.linear_fwd(l.q, l.L1, l.L2, x, out=out, workspace=w)

        def bwd(l, dy, out, w=ws):
            return lambda: binding.linear_bwd_input(l.q, l.L1, l.L2, dy, out=out, workspace=w)

        def qfactors(x, out, backward):
            return lambda: out.copy_(binding.linear_qfactors(square.q, f1, f2, x, backward=backward))

        def grads_from():
            T = binding.linear_intermediate(ws_f, 512, 2560, narrow.q.cfg, R, M, False)
            Tp = binding.linear_intermediate(ws_b, 512, 2560, narrow.q.cfg, R, M, True)
            binding.lora_grads_from(T, Tp, 512, 2560, Y1, Y3, out=(g[2], g[3]), workspace=ws[:256])

        self.calls = [
            fwd(wide, X, Y1),                                        # pair kernel
            fwd(narrow, Y1, Y2),                                     # transposed tiles, reads what the pair kernel wrote
            fwd(square, Y2[:8], s[0][:8]),                           # weight streaming
            bwd(square, s[0][:8], s[1][:8]),
            fwd(plain, s[1][:8], s[2][:8]),                          # no rank-r term: no pre-product in front
            fwd(packed, s[2][:8], s[3][:8]),                         # scales expanded inside the call
            qfactors(s[3][:8], s[4][:8], False),                     # factors dequantized inside the call
            fwd(square, Y2[:100], s[5]),                             # transposed tiles, few rows
            bwd(square, s[5], s[6]),
            fwd(packed, s[6], s[7]),
            qfactors(s[7], s[8], True),
            bwd(plain, s[8], s[9]),
            bwd(narrow, Y2, dY1),                                    # pair kernel
            bwd(wide, dY1, dX1),
            lambda: binding.lora_grads(wide.L1, wide.L2, X, dY1, out=(g[0], g[1]), workspace=ws),
            bwd(narrow, dX1, dY1, ws_b),                             # T', T of the gradients below stay in their workspaces
            fwd(narrow, Y1, Y3, ws_f),                               # writes the dY that the next call reads
            grads_from,
            fwd(square, Y3[:8], s[0][8:16]),                         # streaming behind the weight gradients
            fwd(square, s[0][8:16], X[:8]),                          # and into the first call's input
            fwd(wide, X, Y1),
        ]

    def run(self, synchronize=False):
        self.X.copy_(self.src)
        for t in self.poisoned:
            t.fill_(float("nan"))
        for call in self.calls:
            call()
            if synchronize:
                torch.cuda.synchronize()

    def take(self):
        torch.cuda.synchronize()
        return [t.clone() for t in self.results]


def same_bits(a, b):
    return torch.equal(a.view(torch.int16), b.view(torch.int16))


def test_chained_calls_give_the_bits_of_synchronised_ones():
    chain = Chain()
    chain.run(synchronize=True)
    want = chain.take()
    written = [0, 1, 2, 3, 4] + list(range(5, 19))
    assert all(bool(torch.isfinite(want[i][:8].float()).all()) for i in written)
    for _ in range(20):
        chain.run()
        got = chain.take()
        assert [i for i in written if not same_bits(want[i], got[i])] == []
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        chain.run()
    for _ in range(10):
        for t in chain.poisoned:
            t.fill_(float("nan"))
        graph.replay()
        got = chain.take()
        assert [i for i in written if not same_bits(want[i], got[i])] == []


class EncodeChain:
    """Matrices quantized between other calls: each call reads what the one in front writes, or overwrites what it reads."""

    def __init__(self):
        N, K, rows = 384, 512, 600
        cfgs = [C(3, 64, 8, 256, 32), C(4, 32, 8, 512, 32), C(8, 64, 8, 64, 32), C(2, 16, 4, 64, 16)]      # groups above 256 blocks; packed scales
        W = [torch.from_numpy(inputs.gaussian(9200 + i, (N, K), 0.04)).cuda() for i in range(2)]
        q = [binding.alloc_qmatrix(N, K, c, torch.device("cuda")) for c in cfgs]
        l1b, l2b = inputs.lowrank_factors(9210, N, K, R, 0.02)
        L1, L2 = binding.bf16_from_bits(l1b), binding.bf16_from_bits(l2b)
        X, dY = (binding.bf16_from_bits(inputs.activations(9220 + i, rows, n)) for i, n in enumerate((K, N)))
        ws = torch.empty(max([binding.linear_workspace_bytes(N, K, c, R, m) for c in cfgs for m in (8, rows)] + [binding.packed_sizes(N, K, c)[3] for c in cfgs] +
                             [binding.lora_grads_workspace_bytes(N, K, R, rows)]), dtype=torch.uint8, device="cuda")      # one scratch for all
        g1, g2 = torch.empty(N, R, device="cuda"), torch.empty(R, K, device="cuda")
        qg = binding.alloc_qmatrix(N, R, cfgs[0], torch.device("cuda"))
        Y, Z = (torch.empty(8, rows, N, dtype=torch.bfloat16, device="cuda") for _ in range(2))
        self.results = [Y, Z, g1, g2, qg.codes, qg.scale_codes, qg.scale2.view(torch.uint8)]
        self.codes = torch.empty(4, max(x.codes.numel() for x in q), dtype=torch.uint8, device="cuda")
        self.results.append(self.codes)

        def run():
            for i in range(4):
                binding.encode(W[0], cfgs[i], out=q[i], workspace=ws)
                binding.linear_fwd(q[i], L1, L2, X[:8], out=Y[i, :8], workspace=ws)
                binding.encode(W[1], cfgs[i], out=q[i], workspace=ws)                 # overwrites what the call in front reads
                binding.linear_fwd(q[i], L1, L2, X, out=Y[4 + i], workspace=ws)
                binding.encode(W[0], cfgs[3 - i], out=q[3 - i], workspace=ws)         # two in a row, one scratch
                binding.encode(W[1], cfgs[i], out=q[i], workspace=ws)
                binding.linear_bwd_input(q[i], L1, L2, dY[:4], out=Z[i].view(-1)[:4 * K].view(4, K), workspace=ws)
                binding.lora_grads(L1, L2, X, dY, out=(g1, g2), workspace=ws)
                binding.encode(g1, cfgs[0], out=qg, workspace=ws)                     # a gradient, straight from its kernel
                binding.encode(W[i & 1], cfgs[i], out=q[i], workspace=ws)
                self.codes[i, :q[i].codes.numel()].copy_(q[i].codes)
        self.run = run

    def take(self, run):
        for t in self.results:
            t.view(torch.uint8).fill_(0x5A)
        run()
        torch.cuda.synchronize()
        return [t.view(torch.uint8).clone() for t in self.results]


def test_encodes_between_calls_give_the_bits_of_synchronised_ones(monkeypatch):
    chain = EncodeChain()
    with monkeypatch.context() as m:                  # a synchronisation behind every call of the library
        check, native = binding._check, binding._fast or binding._fast_part()
        m.setattr(binding, "_check", lambda status, where: (check(status, where), torch.cuda.synchronize()))
        m.setattr(binding, "_fast", types.SimpleNamespace(**{name: lambda *a, f=getattr(native, name): (f(*a), torch.cuda.synchronize())[0]
                                                             for name in ("linear", "encode")}))      # (these do not come by _check)
        want = chain.take(chain.run)
    for _ in range(20):
        assert [i for i, (a, b) in enumerate(zip(want, chain.take(chain.run))) if not torch.equal(a, b)] == []
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        chain.run()
    for _ in range(10):
        assert [i for i, (a, b) in enumerate(zip(want, chain.take(graph.replay))) if not torch.equal(a, b)] == []


class PlainChain:
    """Decode-sized calls without a rank-r term on one workspace: a kernel in front of each clears the arrival counters that the one before has
    counted up, and is itself launched while that one ends.  Every result is the next call's input."""

    def __init__(self, rows, b0):
        cfg = C(b0, 64, 8, 64, 32)
        square, wide, narrow = (Layer(9300 + i, N, K, cfg, r=0) for i, (N, K) in enumerate(((1024, 1024), (2048, 1024), (512, 1024))))
        self.layers = [(square, False), (square, True), (wide, False), (wide, True), (narrow, False), (narrow, True), (square, False)] * 3
        for layer, backward in self.layers:
            q = layer.q
            kernel, splits = binding.linear_route(q.N, q.K, cfg, 0, rows, backward)
            if kernel == binding.PATH_STREAM:                    # (the wide matrix's input gradient takes transposed tiles from nine rows on)
                assert splits > 1
            else:
                assert layer is wide and backward and rows > 8
        self.ws = torch.empty(max(binding.linear_workspace_bytes(l.q.N, l.q.K, cfg, 0, rows) for l, _ in self.layers), dtype=torch.uint8, device="cuda")
        self.x = binding.bf16_from_bits(inputs.activations(9310, rows, 1024))
        self.y = [torch.empty(rows, l.q.K if b else l.q.N, dtype=torch.bfloat16, device="cuda") for l, b in self.layers]

    def run(self, synchronize=False):
        x = self.x
        for (layer, backward), y in zip(self.layers, self.y):
            x = (binding.linear_bwd_input if backward else binding.linear_fwd)(layer.q, None, None, x, out=y, workspace=self.ws)
            if synchronize:
                torch.cuda.synchronize()

    def take(self, run, **kwargs):
        for t in self.y:
            t.fill_(float("nan"))
        self.ws.fill_(0x5A)
        run(**kwargs)
        torch.cuda.synchronize()
        assert binding.workspace_status(self.ws) == 0
        return [t.clone() for t in self.y]


@pytest.mark.parametrize("b0", [2, 3, 4, 8])
@pytest.mark.parametrize("rows", [1, 3, 8, 16])
def test_plain_decode_calls_give_the_bits_of_synchronised_ones(rows, b0):
    chain = PlainChain(rows, b0)
    want = chain.take(chain.run, synchronize=True)
    assert all(bool(torch.isfinite(t.float()).all()) and bool((t != 0).any()) for t in want)
    for _ in range(10):
        assert [i for i, (a, b) in enumerate(zip(want, chain.take(chain.run))) if not same_bits(a, b)] == []
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        chain.run()
    for _ in range(5):
        assert [i for i, (a, b) in enumerate(zip(want, chain.take(graph.replay))) if not same_bits(a, b)] == []


@pytest.mark.parametrize("b0,rows", [(3, 48), (8, 40), (2, 300)])
def test_a_matrix_encoded_in_front_of_a_plain_call(b0, rows):
    """Transposed tiles without a rank-r term are the first kernel of their call: copies of the codes, loads of the scales and copies of the
    activations wait for the encoder, and for the call that wrote the activations."""
    cfg, N, K = C(b0, 64, 8, 64, 32), 768, 768
    W = [torch.from_numpy(inputs.gaussian(9400 + i, (N, K), 0.04)).cuda() for i in range(3)]
    q = binding.alloc_qmatrix(N, K, cfg, torch.device("cuda"))
    assert binding.linear_path(N, K, cfg, 0, rows, False) == binding.PATH_TC_ONE
    ws = torch.empty(max(binding.linear_workspace_bytes(N, K, cfg, 0, rows), binding.packed_sizes(N, K, cfg)[3]), dtype=torch.uint8, device="cuda")
    x = binding.bf16_from_bits(inputs.activations(9410, rows, K))
    ys = [torch.empty(rows, N, dtype=torch.bfloat16, device="cuda") for _ in range(9)]

    def run(synchronize=False):
        sync = torch.cuda.synchronize if synchronize else lambda: None
        a = x
        for i, y in enumerate(ys):
            binding.encode(W[i % 3], cfg, out=q, workspace=ws)
            sync()
            a = (binding.linear_bwd_input if i % 2 else binding.linear_fwd)(q, None, None, a, out=y, workspace=ws)
            sync()
        torch.cuda.synchronize()
        return [y.clone() for y in ys]

    want = run(synchronize=True)
    assert all(bool(torch.isfinite(t.float()).all()) and bool((t != 0).any()) for t in want)
    for _ in range(10):
        for y in ys:
            y.fill_(float("nan"))
        assert [i for i, (a, b) in enumerate(zip(want, run())) if not same_bits(a, b)] == []
