"""GPU check of the K pass of the bf16 stored route around its blocks of 32 sequences: whole numbers small enough for every step to be
exact (bf16 gradients, float32 sums), so K has to be what int64 gives, to the bit."""

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def b():
    from paper_2512_23353_b200 import binding
    return binding


def _case(B, L, d_in, d_outs, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    off = np.arange(B + 1, dtype=np.int64) * L
    draw = lambda d: torch.randint(-1, 2, (B * L, d), device="cuda", generator=gen)  # noqa: E731
    X, dYs = draw(d_in), [draw(o) for o in d_outs]
    Ks = []
    for dY in dYs:
        G = (dY.view(B, L, -1, 1) * X.view(B, L, 1, -1)).sum(1).reshape(B, -1).double()
        assert G.abs().max() <= 256
        Ks.append((G @ G.T).float())
    return X.bfloat16(), [dY.bfloat16() for dY in dYs], off, Ks


@pytest.mark.parametrize("B", [1, 2, 3, 4, 5, 7, 8, 9, 13, 16, 17, 20, 31, 32, 33, 35, 63, 64, 65, 96, 97, 127, 128, 129, 144, 145, 160, 161, 193, 255, 256])
@pytest.mark.parametrize("L,d_in,d_out", [(1, 72, 40), (2, 264, 296)])
def test_exact(b, B, L, d_in, d_out):
    X, (dY,), off, (want,) = _case(B, L, d_in, [d_out], 1000 * B + d_in)
    raw = torch.full((B * B + 3,), float("nan"), device="cuda")
    for shift in (0, 1, 3):  # K may start at any element
        K = raw[shift:shift + B * B].view(B, B)
        ws = b.alloc_workspace(b.BF16, B * L, d_in, d_out, B, b.PATH_MATERIALISE)
        ws.fill_(0xFF)
        info = torch.zeros(1, dtype=torch.int32, device="cuda")
        for _ in range(2):  # the second pass finds the first one's sums
            b.isopo_layer_gram(X, dY, off, K, ws, info, b.PATH_MATERIALISE)
        torch.cuda.synchronize()
        assert int(info.item()) == 0
        assert torch.equal(K, want)


@pytest.mark.parametrize("B", [30, 31, 200])
def test_exact_shared_input(b, B):
    """Projections of which one would complete K in its last CTA and another would not."""
    d_outs = [8, 600, 256]
    X, dYs, off, want = _case(B, 2, 520, d_outs, B)
    ws = [b.alloc_workspace(b.BF16, 2 * B, 520, o, B, b.PATH_MATERIALISE) for o in d_outs]
    Ks = [torch.full((B, B), float("nan"), device="cuda") for _ in d_outs]
    info = torch.zeros(1, dtype=torch.int32, device="cuda")
    b.isopo_layer_gram_shared_x_stored(X, dYs, off, Ks, ws, info)
    torch.cuda.synchronize()
    assert int(info.item()) == 0
    for K, w in zip(Ks, want):
        assert torch.equal(K, w)


@pytest.mark.parametrize("B,d_in,d_out,n", [(40, 512, 640, 148), (64, 512, 640, 148), (100, 512, 320, 148), (128, 512, 320, 148),
                                            (160, 512, 160, 148), (256, 512, 160, 148), (64, 896, 128, 56), (100, 896, 128, 112),
                                            (20, 512, 512, 64), (32, 512, 512, 64)])
def test_one_addition_per_cta(b, B, d_in, d_out, n):
    """K of gradients of one sign, exact in bf16, is a sum of up to n positive float32 additions, one per CTA of eight boxes or more.
    Rounding an addition to S errs by ulp(S) / sqrt(12), ulp(S)^2 is 0.54 * 2^-46 S^2 in the mean, and S grows evenly: n additions leave
    2^-23 sqrt(0.015 n) of the result, 1.78e-7 for 148 and 2.5e-7 for two of each; 18 % are left for the tensor cores' own sums (few here)
    and what they err by in all entries alike is taken out."""
    errors = []
    for seed in range(4):
        gen = torch.Generator(device="cuda")
        gen.manual_seed(1000 * B + seed)
        X, dY = (torch.randint(8, 16, (B, d), device="cuda", generator=gen).bfloat16() for d in (d_in, d_out))
        want = (X.double() @ X.double().T) * (dY.double() @ dY.double().T)
        off = np.arange(B + 1, dtype=np.int64)
        ws = b.alloc_workspace(b.BF16, B, d_in, d_out, B, b.PATH_MATERIALISE)
        K, info = torch.empty((B, B), device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")
        for _ in range(3):
            b.isopo_layer_gram(X, dY, off, K, ws, info, b.PATH_MATERIALISE)
            e = (K.double() - want) / want
            errors.append((e - e.mean()).pow(2).mean().sqrt().item())
        assert int(info.item()) == 0
    assert np.mean(errors) <= 1.18 * 2.0 ** -23 * (0.015 * n) ** 0.5
