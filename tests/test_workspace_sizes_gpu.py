"""bf16 workspaces without the areas that only make the kernels faster (operands at whole lines, padded sums of the K pass): what the
offsets, the token map, the scaled operand and the gradients take serves every call, a byte less is refused, and the results are
those of a full workspace up to the order of float32 sums (K, F2) and the rounding of the scaled operand to bf16 (dW: 2^-8 of a product)."""

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def b():
    from paper_2512_23353_b200 import binding
    return binding


def _up(n):
    return -(-n // 1024) * 1024


def _ws(n):
    raw = torch.zeros(n + 1024, dtype=torch.uint8, device="cuda")
    return raw[(-raw.data_ptr()) % 1024:][:n]


def _rel(a, c):
    return ((a.double() - c.double()).norm() / c.double().norm()).item()


# (lengths, d_in, d_out, stored): copies of both operands and of one, narrow operand at lines, no room for the sums of 40 and 200 sequences
@pytest.mark.parametrize("Ls,d_in,d_out,stored", [([30] * 50, 1080, 312, False), ([500] * 3, 136, 2368, False), ([9] * 11, 264, 2504, False),
                                                  ([3] * 40, 200, 264, True), ([2] * 200, 128, 136, True), ([300] * 40, 200, 264, True)])
def test_least_workspace(b, Ls, d_in, d_out, stored):
    off, B, T = np.concatenate([[0], np.cumsum(Ls)]).astype(np.int64), len(Ls), sum(Ls)
    path = b.PATH_MATERIALISE if stored else b.PATH_GRAM
    gen = torch.Generator(device="cuda")
    gen.manual_seed(T)
    X, dY = (torch.randn((T, d), device="cuda", generator=gen).bfloat16() for d in (d_in, d_out))
    c = torch.randn(B, device="cuda", generator=gen)
    least = 1024 + _up(8 * (B + 1)) + _up(4 * T)
    least += _up(8 * B) + _up(2 * B * (-(-d_out // 32) * 32) * d_in) if stored else _up(2 * T * min(d_in, d_out))
    full = b.isopo_workspace_bytes(b.BF16, T, d_in, d_out, B, path)
    assert full > least or T >= B * B
    got = []
    between = [least + 1024 + 1000, (least + full) // 2 + 1, full - 1] if full > least + 4096 else []  # fewer copies, or none
    for n in (full, least, *between):
        K, dW, info = torch.empty((B, B), device="cuda"), torch.empty((d_out, d_in), device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")
        raw = _ws(n + 4096)
        raw[n:] = 77
        ws = raw[:n]
        b.isopo_layer_gram(X, dY, off, K, ws, info, path)
        b.isopo_weight_grad(X, dY, c, off, dW, ws, info, path)
        torch.cuda.synchronize()
        assert int(info.item()) == 0
        assert (raw[n:] == 77).all()  # nothing behind it is written
        got.append((K, dW))
    for K, dW in got[1:]:
        assert _rel(K, got[0][0]) <= 2e-6 and _rel(dW, got[0][1]) <= 2.0 ** -8
    with pytest.raises(Exception):
        b.isopo_layer_gram(X, dY, off, K, _ws(least - 1024), info, path)
    with pytest.raises(Exception):
        b.isopo_weight_grad(X, dY, c, off, dW, _ws(least - 1024), info, path)


@pytest.mark.parametrize("Ls,d_in,d_out,n", [([400] * 3, 1080, 312, 40), ([30] * 3, 200, 1032, 130)])
def test_least_sampled_workspace(b, Ls, d_in, d_out, n):
    off, B, T = np.concatenate([[0], np.cumsum(Ls)]).astype(np.int64), len(Ls), sum(Ls)
    X, dY = (torch.randn((T, d), device="cuda").bfloat16() for d in (d_in, d_out))
    rows = np.random.default_rng(n).choice(T, n, replace=n > T).astype(np.int64)
    least = 1024 + _up(8 * (B + 1)) + _up(4 * T) + _up(2 * T * min(d_in, d_out)) + _up(2 * n * d_in) + _up(2 * n * d_out) + _up(4 * n * B) + 1024
    full = b.isopo_sampled_workspace_bytes(b.BF16, T, d_in, d_out, B, n)
    assert full > least
    A, got = torch.ones(B, device="cuda"), []
    for size in (full, least):
        c, F2, info = torch.empty(B, device="cuda"), torch.empty(B, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")
        dW, ws = torch.empty((d_out, d_in), device="cuda"), _ws(size)
        b.isopo_sampled_coefficients(X, dY, off, rows, A, 0.0, c, ws, info, F2)
        b.isopo_weight_grad(X, dY, c, off, dW, ws, info, b.PATH_GRAM)
        torch.cuda.synchronize()
        assert int(info.item()) == 0
        got.append((F2, dW))
    assert _rel(got[1][0], got[0][0]) <= 2e-6 and _rel(got[1][1], got[0][1]) <= 2.0 ** -8
    with pytest.raises(Exception):
        b.isopo_sampled_coefficients(X, dY, off, rows, A, 0.0, c, _ws(least - 1024), info, F2)
