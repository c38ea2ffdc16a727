"""Passes enqueued back to back, nothing waiting in between: every kernel may be set up while the one before it runs, and
must not touch memory before everything ahead of it is done.  Two layers of different sizes take turns on one workspace and
one set of outputs, so a kernel that ran early would read or clear the other layer's data; the outputs of the last pass of
each are compared with those of a pass on an idle device.  Also the sizes at which offsets and sample rows change the way
they travel to the device (383 / 384 and 2047 / 2048 sequences, 256 / 257 samples).

Bounds: only the order of float32 atomic additions differs between passes: 2e-6 on K and F^2; dW of the pre-scaled route
inherits coefficients that may differ in their last bit, which flips bf16 roundings of single operand elements: 3e-4."""

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def b():
    from paper_2512_23353_b200 import binding
    return binding


class Layer:
    def __init__(self, b, dtype, lens, d_in, d_out, seed):
        g = torch.Generator(device="cuda").manual_seed(seed)
        self.off = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
        self.T, self.B, self.d_in, self.d_out = int(self.off[-1]), len(lens), d_in, d_out
        self.code = b.BF16 if dtype == torch.bfloat16 else b.F32
        self.X = torch.randn(self.T, d_in, device="cuda", generator=g).to(dtype)
        self.dY = (0.1 * torch.randn(self.T, d_out, device="cuda", generator=g)).to(dtype)
        self.A = torch.randn(self.B, device="cuda", generator=g)

    def run(self, b, buf, path):
        K, c = buf["K"][:self.B * self.B], buf["c"][:self.B]
        dW = buf["dW"][:self.d_out * self.d_in].view(self.d_out, self.d_in)
        b.isopo_layer_gram(self.X, self.dY, self.off, K, buf["ws"], buf["info"], path)
        b.isopo_transform_advantages(K, self.A, b.VAR_NORMALISED, 1e-3, c, buf["info"])
        b.isopo_weight_grad(self.X, self.dY, c, self.off, dW, buf["ws"], buf["info"], path, 0.0)
        return K, c, dW


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("route", ["gram", "stored"])
def test_two_layers_take_turns(b, dtype, route):
    path = b.PATH_GRAM if route == "gram" else b.PATH_MATERIALISE
    layers = [Layer(b, dtype, [40, 1, 300, 77], 264, 136, 1), Layer(b, dtype, [5 + i % 9 for i in range(60)], 128, 520, 2)]
    n = max(b.isopo_workspace_bytes(l.code, l.T, l.d_in, l.d_out, l.B, path) for l in layers)
    raw = torch.empty(n + 1024, dtype=torch.uint8, device="cuda")
    shift = (-raw.data_ptr()) % 1024
    buf = {"ws": raw[shift:shift + n], "K": torch.empty(3600, device="cuda"), "c": torch.empty(60, device="cuda"),
           "dW": torch.empty(128 * 520, device="cuda"), "info": torch.zeros(1, dtype=torch.int32, device="cuda")}
    want = []
    for l in layers:
        torch.cuda.synchronize()
        out = l.run(b, buf, path)
        torch.cuda.synchronize()
        want.append([t.clone() for t in out])
    for i in range(40):
        for l, w in zip(layers, want):
            got = l.run(b, buf, path)
            if i % 8 == 7:
                for g, q, tol in zip(got, w, (2e-6, 2e-6, 3e-4)):
                    assert float((g - q).norm() / q.norm()) <= tol
    assert int(buf["info"].item()) == 0


@pytest.mark.parametrize("B", [382, 383, 384, 2046, 2047, 2048, 2049])
def test_offsets_of_many_sequences(b, B):
    """Sequences of one token, two projected widths: K is (dY dY^T) o (X X^T), dW = (c dY)^T X."""
    l = Layer(b, torch.float32, [1] * B, 20, 12, B)
    ws = b.alloc_workspace(b.F32, l.T, 20, 12, B, b.PATH_GRAM)
    buf = {"ws": ws, "K": torch.empty(B * B, device="cuda"), "c": torch.empty(B, device="cuda"),
           "dW": torch.empty(240, device="cuda"), "info": torch.zeros(1, dtype=torch.int32, device="cuda")}
    K, c, dW = l.run(b, buf, b.PATH_GRAM)
    X, dY = l.X.double(), l.dY.double()
    want = (dY @ dY.T) * (X @ X.T)
    assert float((K.view(B, B).double() - want).norm() / want.norm()) <= 2e-6
    dW_want = (c.double()[:, None] * dY).T @ X
    assert float((dW.double() - dW_want).norm() / dW_want.norm()) <= 2e-6


@pytest.mark.parametrize("n", [255, 256, 257, 4096])
def test_sample_rows(b, n):
    l = Layer(b, torch.float32, [900, 2300, 1000], 24, 16, n)
    rows = np.random.default_rng(n).permutation(l.T)[:n].astype(np.int64)
    ws = b.alloc_sampled_workspace(b.F32, l.T, 24, 16, 3, n)
    c, F2, info = torch.empty(3, device="cuda"), torch.empty(3, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")
    b.isopo_sampled_coefficients(l.X, l.dY, l.off, rows, l.A, 0.0, c, ws, info, F2)
    X, dY = l.X.double(), l.dY.double()
    a0, g0 = X[rows], dY[rows]
    M = ((g0 @ dY.T) * (a0 @ X.T))
    M = torch.stack([M[:, l.off[i]:l.off[i + 1]].sum(1) for i in range(3)], 1)
    want = (M ** 2).sum(0) / (a0.pow(2).sum(1) * g0.pow(2).sum(1)).sum()
    assert float((F2.double() - want).norm() / want.norm()) <= 4e-6


@pytest.mark.parametrize("route", ["gram", "stored"])
@pytest.mark.parametrize("B,d_in,d_out", [(1, 40, 24), (18, 40, 24), (15, 40, 24), (16, 40, 24), (17, 40, 24), (32, 40, 24), (33, 40, 24),
                                          (17, 384, 512), (32, 384, 512)])
def test_k_is_completed(b, route, B, d_in, d_out):
    """Few sequences and little work: the only or the last CTA of the kernel completes K, otherwise a kernel of its own does.  Bounds:
    (d_in + d_out) 2^-23, the sum of the two accumulations' worst relative errors; stored gradients are rounded to bf16, 2^-9
    for each of the two factors."""
    l = Layer(b, torch.bfloat16, [1 + 3 * (i % 5) for i in range(B)], d_in, d_out, B)
    path = b.PATH_GRAM if route == "gram" else b.PATH_MATERIALISE
    buf = {"ws": b.alloc_workspace(l.code, l.T, d_in, d_out, B, path), "K": torch.empty(B * B, device="cuda"),
           "info": torch.zeros(1, dtype=torch.int32, device="cuda")}
    X, dY = l.X.double(), l.dY.double()
    G = torch.stack([dY[l.off[i]:l.off[i + 1]].T @ X[l.off[i]:l.off[i + 1]] for i in range(B)]).flatten(1)
    want = G @ G.T
    tol = (d_in + d_out) * 2.0 ** -23 + (2.0 ** -8 if route == "stored" else 0.0)
    for _ in range(3):  # the counter starts anew in every pass
        buf["K"].fill_(float("nan"))
        b.isopo_layer_gram(l.X, l.dY, l.off, buf["K"], buf["ws"], buf["info"], path)
        got = buf["K"].view(B, B)
        assert torch.equal(got, got.T)
        assert float((got.double() - want).norm() / want.norm()) <= tol
    assert int(buf["info"].item()) == 0


@pytest.mark.parametrize("B", [383, 384, 2047, 2048])
def test_offsets_of_the_scaling_pass(b, B):
    """dW of one-token sequences: (bf16(c dY))^T X.  The reference rounds c dY the same way, so only the accumulation differs:
    T 2^-23 at worst, taken as 1e-5 of the norm."""
    l = Layer(b, torch.bfloat16, [1] * B, 256, 256, B)
    ws = b.alloc_workspace(b.BF16, l.T, 256, 256, B, b.PATH_GRAM)
    c = torch.randn(B, device="cuda", generator=torch.Generator(device="cuda").manual_seed(B))
    dW, info = torch.empty(256, 256, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")
    b.isopo_weight_grad(l.X, l.dY, c, l.off, dW, ws, info, b.PATH_GRAM, 0.0)
    want = (c[:, None] * l.dY.float()).bfloat16().double().T @ l.X.double()
    assert float((dW.double() - want).norm() / want.norm()) <= 1e-5
    assert int(info.item()) == 0
