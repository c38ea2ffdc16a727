"""Token-Gram kernel with 2-CTA tiles (256 x 256 tokens): wide layers from 2049 tokens on, with an odd and an even
number of 128-token tiles, ragged last tiles, feature counts that end inside a 64-feature step, and sequences that are shorter
than a group of 32 columns, that end on a tile's edge and that span tiles; and the widths beside the line to the 1-CTA kernel.

Reference: K = S^T ((X X^T) o (dY dY^T)) S in float64, S the token -> sequence matrix.  Bound: (d_in + d_out) 2^-24, the worst
relative error of the two accumulations."""

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,d_in,d_out", [(2049, 2560, 2568), (2176, 2560, 2560), (2177, 5000, 136), (2303, 136, 5000), (2560, 2568, 2560),
                                          (3841, 1536, 1528), (9600, 512, 88), (9601, 512, 136), (5120, 640, 640), (5120, 128, 8)])
@pytest.mark.parametrize("law", ["short", "long"])
def test_gram_pair(T, d_in, d_out, law):
    from paper_2512_23353_b200 import binding as b
    rng = np.random.default_rng(T + d_in)
    if law == "short":
        cuts = np.unique(np.concatenate([[0, 1, 31, 32, 128, 256], rng.integers(1, T, 150), [T - 1, T]]))
    else:
        cuts = np.array([0, 128, 640, 1500, T])
    off, B = cuts.astype(np.int64), len(cuts) - 1
    g = torch.Generator(device="cuda").manual_seed(T)
    X = torch.randn(T, d_in, device="cuda", generator=g).bfloat16()
    dY = torch.randn(T, d_out, device="cuda", generator=g).bfloat16()
    S = torch.zeros(T, B, device="cuda", dtype=torch.float64)
    S[torch.arange(T, device="cuda"), torch.from_numpy(np.repeat(np.arange(B), np.diff(off))).cuda()] = 1
    want = S.T @ ((X.double() @ X.double().T) * (dY.double() @ dY.double().T)) @ S
    K, info = torch.full((B * B,), float("nan"), device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")
    ws = b.alloc_workspace(b.BF16, T, d_in, d_out, B, b.PATH_GRAM)
    b.isopo_layer_gram(X, dY, off, K, ws, info, b.PATH_GRAM)
    got = K.view(B, B).double()
    assert torch.equal(got, got.T)
    assert float((got - want).norm() / want.norm()) <= (d_in + d_out) * 2.0 ** -24
    assert int(info.item()) == 0


@pytest.mark.parametrize("T,d_in,d_outs", [(2049, 2560, [2568, 136]), (3841, 1536, [1536, 256, 256]), (5121, 136, [2560, 64, 1000]),
                                           (2560, 2560, [2560]), (4000, 896, [896, 128, 128])])
@pytest.mark.parametrize("law", ["short", "long"])
def test_gram_pair_shared(T, d_in, d_outs, law):
    """Projections that share X: P stays in registers while their Q take turns in tensor memory."""
    from paper_2512_23353_b200 import binding as b
    rng = np.random.default_rng(T)
    cuts = np.unique(np.concatenate([[0, 1, 31, 160], rng.integers(1, T, 120), [T]])) if law == "short" else np.array([0, 700, 1024, T])
    off, B, n = cuts.astype(np.int64), len(cuts) - 1, len(d_outs)
    g = torch.Generator(device="cuda").manual_seed(T)
    X = torch.randn(T, d_in, device="cuda", generator=g).bfloat16()
    dYs = [torch.randn(T, d, device="cuda", generator=g).bfloat16() for d in d_outs]
    S = torch.zeros(T, B, device="cuda", dtype=torch.float64)
    S[torch.arange(T, device="cuda"), torch.from_numpy(np.repeat(np.arange(B), np.diff(off))).cuda()] = 1
    Ks, info = [torch.full((B, B), float("nan"), device="cuda") for _ in d_outs], torch.zeros(1, dtype=torch.int32, device="cuda")
    ws = b.alloc_workspace(b.BF16, T, d_in, max(d_outs), B, b.PATH_GRAM)
    for _ in range(2):
        b.isopo_layer_gram_shared_x(X, dYs, off, Ks, ws, info)
    P = X.double() @ X.double().T
    for dY, K, d_out in zip(dYs, Ks, d_outs):
        want = S.T @ (P * (dY.double() @ dY.double().T)) @ S
        assert torch.equal(K, K.T)
        assert float((K.double() - want).norm() / want.norm()) <= (d_in + d_out) * 2.0 ** -24
    assert int(info.item()) == 0
