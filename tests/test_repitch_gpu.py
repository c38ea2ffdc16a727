"""GPU parity of the Gram route around the copies of its operands at a pitch of whole 128-byte lines (1000 tokens on, widths off the
64-column grid, up to 2047 sequences), against torch float64 on the same bf16 inputs: 1e-5 in norm, as the kernels give without them."""

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu
TOL = 1e-5


@pytest.fixture(scope="module")
def b():
    from paper_2512_23353_b200 import binding
    return binding


def _inputs(off, d_in, d_outs):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(off[-1]) + d_in)
    T = int(off[-1])
    shared = torch.randn((T, 2), device="cuda", generator=gen)
    make = lambda d: (torch.randn((T, d), device="cuda", generator=gen) + shared @ torch.randn((2, d), device="cuda", generator=gen)).bfloat16()  # noqa: E731
    return make(d_in), [make(o) for o in d_outs]


def _want(X, dY, off):
    B, T = len(off) - 1, X.shape[0]
    seq = torch.from_numpy(np.repeat(np.arange(B), np.diff(off))).cuda()
    pairs = (dY.double() @ dY.double().T) * (X.double() @ X.double().T)
    rows = torch.zeros((B, T), dtype=torch.float64, device="cuda").index_add_(0, seq, pairs)
    return torch.zeros((B, B), dtype=torch.float64, device="cuda").index_add_(1, seq, rows)


@pytest.mark.parametrize("T,B,d_in,d_outs", [
    (999, 20, 72, [136]), (1000, 20, 72, [136]), (1000, 20, 128, [136]), (1000, 20, 72, [128]), (1003, 7, 8, [8]),
    (2500, 383, 328, [264]), (2500, 384, 328, [264]), (2500, 2047, 200, [72]), (2500, 2048, 200, [72]),
    (3001, 90, 1032, [520, 264, 72]),   # projections that share X: room for the copies of X and of the widest
    (1500, 30, 1024, [72, 520, 520]), (1500, 30, 72, [512, 64, 8])])
def test_gram(b, T, B, d_in, d_outs):
    off = np.concatenate([[0], np.sort(np.random.default_rng(T + B).choice(np.arange(1, T), B - 1, replace=False)), [T]]).astype(np.int64)
    X, dYs = _inputs(off, d_in, d_outs)
    before = [t.clone() for t in [X, *dYs]]
    ws = [b.alloc_workspace(b.BF16, T, d_in, o, B, b.PATH_GRAM) for o in d_outs]
    wide = max(ws, key=lambda w: w.numel())
    wide.fill_(0xFF)
    info = torch.zeros(1, dtype=torch.int32, device="cuda")
    Ks = [torch.full((B, B), float("nan"), device="cuda") for _ in dYs]
    if len(dYs) > 1:
        b.isopo_layer_gram_shared_x(X, dYs, off, Ks, wide, info)
    else:
        b.isopo_layer_gram(X, dYs[0], off, Ks[0], wide, info, b.PATH_GRAM)
    torch.cuda.synchronize()
    assert int(info.item()) == 0
    for K, dY in zip(Ks, dYs):
        want = _want(X, dY, off)
        assert ((K.double() - want).norm() / want.norm()).item() <= TOL
        assert torch.equal(K, K.T)
    assert all(torch.equal(a, t) for a, t in zip(before, [X, *dYs]))
    # the scaled operand of the weight gradient lies at such a pitch too: whole numbers small enough for every step to be exact
    X, dY, c = (torch.randint(-n, n + 1, shape, device="cuda") for n, shape in [(1, X.shape), (1, dYs[0].shape), (8, (B,))])
    rows = c[torch.from_numpy(np.repeat(np.arange(B), np.diff(off))).cuda()][:, None]
    want = (rows.double() * dY.double()).T @ X.double()
    for beta in (0.0, 1.0):
        dW = torch.full((d_outs[0], d_in), 500.0 if beta else float("nan"), device="cuda")
        b.isopo_weight_grad(X.bfloat16(), dY.bfloat16(), c.float(), off, dW, ws[0], info, b.PATH_GRAM, beta)
        assert torch.equal(dW.double(), want + 500.0 * beta)
