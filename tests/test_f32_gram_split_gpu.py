"""float32 token-Gram kernel and sampled estimator where several CTAs share a tile's features: against torch float64.  P and Q are
float32 sums over up to 4096 features (a fraction of 2^-24 each in norm, since partial sums meet), the rest is float64: 2e-6, as for
the other float32 kernels."""

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu
TOL = 2e-6


@pytest.fixture(scope="module")
def b():
    from paper_2512_23353_b200 import binding
    return binding


def _inputs(Ls, d_in, d_out, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    off = np.concatenate([[0], np.cumsum(Ls)]).astype(np.int64)
    T = int(off[-1])
    make = lambda d: torch.randn((T, d), device="cuda", generator=gen) + torch.randn(d, device="cuda", generator=gen)  # noqa: E731
    return off, make(d_in), make(d_out)


# one, two, four and eight CTAs to a tile of 32, one and two to a tile of 64; odd widths; shares of X alone, of both, of dY alone
@pytest.mark.parametrize("Ls,d_in,d_out", [
    ([1], 300, 41), ([31, 1], 1000, 3), ([5, 28], 7, 1030), ([3] * 30, 129, 515), ([70, 80, 90, 60], 896, 896),
    ([200, 150, 1], 300, 1300), ([7] * 100, 251, 1121), ([30] * 31, 296, 577), ([64] * 19, 1024, 1030), ([64] * 24, 512, 2000)])
def test_gram(b, Ls, d_in, d_out):
    off, X, dY = _inputs(Ls, d_in, d_out, d_in + d_out)
    B, T = len(Ls), int(off[-1])
    ws = b.alloc_workspace(b.F32, T, d_in, d_out, B, b.PATH_GRAM)
    K, info = torch.empty((B, B), device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")
    b.isopo_layer_gram(X, dY, off, K, ws, info, b.PATH_GRAM)
    torch.cuda.synchronize()
    assert int(info.item()) == 0
    seq = torch.from_numpy(np.repeat(np.arange(B), Ls)).cuda()
    pairs = (X.double() @ X.double().T) * (dY.double() @ dY.double().T)
    want = torch.zeros((B, T), dtype=torch.float64, device="cuda").index_add_(0, seq, pairs)
    want = torch.zeros((B, B), dtype=torch.float64, device="cuda").index_add_(1, seq, want)
    assert ((K.double() - want).norm() / want.norm()).item() <= TOL
    assert torch.equal(K, K.T)


@pytest.mark.parametrize("Ls,d_in,d_out,n", [([40, 88], 712, 1169, 128), ([100, 150, 30], 1536, 1539, 32), ([500, 438], 1539, 185, 128),
                                             ([3] * 400, 251, 617, 33), ([700] * 10, 1481, 1513, 128), ([10], 2048, 2048, 1)])
def test_sampled(b, Ls, d_in, d_out, n):
    off, X, dY = _inputs(Ls, d_in, d_out, d_in + n)
    B, T = len(Ls), int(off[-1])
    rows = np.random.default_rng(n).permutation(T)[:n].astype(np.int64)
    raw = torch.empty(b.isopo_sampled_workspace_bytes(b.F32, T, d_in, d_out, B, n) + 1024, dtype=torch.uint8, device="cuda")
    ws, info = raw[(-raw.data_ptr()) % 1024:], torch.zeros(1, dtype=torch.int32, device="cuda")
    A, c, F2 = torch.ones(B, device="cuda"), torch.empty(B, device="cuda"), torch.empty(B, device="cuda")
    b.isopo_sampled_coefficients(X, dY, off, rows, A, 0.0, c, ws, info, F2)
    torch.cuda.synchronize()
    assert int(info.item()) == 0
    x, y, r = X.double(), dY.double(), torch.from_numpy(rows).cuda()
    seq = torch.from_numpy(np.repeat(np.arange(B), Ls)).cuda()
    M = torch.zeros((n, B), dtype=torch.float64, device="cuda").index_add_(1, seq, (y[r] @ y.T) * (x[r] @ x.T))
    want = (M ** 2).sum(0) / ((y[r] ** 2).sum(1) * (x[r] ** 2).sum(1)).sum()
    assert ((F2.double() - want).norm() / want.norm()).item() <= 2 * TOL  # squares


# tiles of 64 by two CTAs: one of them without a feature of X, without one of dY, its first stage the first of dY's
@pytest.mark.parametrize("Ls,d_in,d_out", [([20] * 35, 48, 3000), ([350, 351], 3000, 48), ([64] * 11, 1536, 1536), ([50] * 24, 893, 899)])
def test_gram_wide_tiles_by_two(b, Ls, d_in, d_out):
    test_gram(b, Ls, d_in, d_out)


# 32 samples leave half of a tile of 64 empty; 65 take tiles of 64; two CTAs to a tile
@pytest.mark.parametrize("Ls,d_in,d_out,n", [([999] * 8, 448, 448, 32), ([999] * 8, 448, 450, 65), ([250] * 8, 896, 896, 128)])
def test_sampled_tiles(b, Ls, d_in, d_out, n):
    test_sampled(b, Ls, d_in, d_out, n)
