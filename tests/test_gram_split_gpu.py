"""GPU parity of K and of the sampled estimator for few tokens, where a cluster of CTAs shares the features of a tile: against
torch float64 on the same bf16 inputs.  Products of bf16 numbers are exact in float32; a sum over 128 x 128 token pairs of float32
sums over up to 14,336 features stays within 1e-5 in norm (observed 2e-7 to 1e-6)."""

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu
TOL = 1e-5


@pytest.fixture(scope="module")
def b():
    from paper_2512_23353_b200 import binding
    return binding


def _inputs(Ls, d_in, d_outs, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    off = np.concatenate([[0], np.cumsum(Ls)]).astype(np.int64)
    T = int(off[-1])
    shared = torch.randn((T, 2), device="cuda", generator=gen)  # overlaps between sequences
    make = lambda d: (torch.randn((T, d), device="cuda", generator=gen) + shared @ torch.randn((2, d), device="cuda", generator=gen)).bfloat16()  # noqa: E731
    return off, make(d_in), [make(o) for o in d_outs]


def _want(X, dY, off):
    B = len(off) - 1
    S = torch.zeros((B, X.shape[0]), dtype=torch.float64, device="cuda")
    for i in range(B):
        S[i, off[i]:off[i + 1]] = 1.0
    return S @ ((dY.double() @ dY.double().T) * (X.double() @ X.double().T)) @ S.T


# two, four and eight CTAs to a tile; one tile and several; a share with features of X and of dY, and none such
CASES = [
    ([1], 768, [768]),
    ([100, 27], 896, [896]),
    ([64, 1, 63], 1536, [1536]),             # one tile exactly; sequences on both sides of 32 rows
    ([4] * 33, 3072, [3072]),                # a second tile of four tokens; the other triangle by a kernel of its own
    ([3] * 40, 72, [4096]),
    ([50, 60, 70, 80, 90], 4096, [8]),
    ([30] * 30, 2048, [2056]),               # 36 tiles: two CTAs
    ([5, 250, 1, 1, 200], 1000, [6400]),
    ([40, 45, 60], 1024, [1024, 256, 264]),  # projections that share X
    ([150, 300], 896, [4864, 4872]),
]


@pytest.mark.parametrize("Ls,d_in,d_outs", CASES)
def test_gram(b, Ls, d_in, d_outs):
    off, X, dYs = _inputs(Ls, d_in, d_outs, 3 * d_in + d_outs[0])
    B, T = len(Ls), int(off[-1])
    info = torch.zeros(1, dtype=torch.int32, device="cuda")
    Ks = [torch.full((B, B), float("nan"), device="cuda") for _ in dYs]
    ws = [b.alloc_workspace(b.BF16, T, d_in, o, B, b.PATH_GRAM) for o in d_outs]
    if len(dYs) > 1:
        b.isopo_layer_gram_shared_x(X, dYs, off, Ks, max(ws, key=lambda w: w.numel()), info)
    else:
        b.isopo_layer_gram(X, dYs[0], off, Ks[0], ws[0], info, b.PATH_GRAM)
    torch.cuda.synchronize()
    assert int(info.item()) == 0
    for K, dY in zip(Ks, dYs):
        want = _want(X, dY, off)
        err = ((K.double() - want).norm() / want.norm()).item()
        print(f"T={T} B={B} {d_in}->{dY.shape[1]} rel {err:.1e}")
        assert err <= TOL
        assert torch.equal(K, K.T)


@pytest.mark.parametrize("Ls,d_in,d_out,n", [([40, 48], 2160, 416, 88), ([1, 200, 7], 896, 896, 1), ([300] * 20, 512, 2360, 128),
                                             ([90, 400], 1024, 1024, 300),
                                             ([700] * 30, 512, 520, 9), ([700] * 30, 512, 520, 33), ([40, 48], 2160, 416, 7)])  # boxes of fewer rows
def test_sampled(b, Ls, d_in, d_out, n):
    off, X, (dY,) = _inputs(Ls, d_in, [d_out], 5 * d_in + n)
    B, T = len(Ls), int(off[-1])
    rows = np.random.default_rng(n).permutation(T)[:n].astype(np.int64)
    ws = torch.empty(b.isopo_sampled_workspace_bytes(b.BF16, T, d_in, d_out, B, n) + 1024, dtype=torch.uint8, device="cuda")
    ws = ws[(-ws.data_ptr()) % 1024:]
    info = torch.zeros(1, dtype=torch.int32, device="cuda")
    A, c, F2 = torch.ones(B, device="cuda"), torch.empty(B, device="cuda"), torch.empty(B, device="cuda")
    b.isopo_sampled_coefficients(X, dY, off, rows, A, 0.0, c, ws, info, F2)
    torch.cuda.synchronize()
    assert int(info.item()) == 0
    x, y = X.double(), dY.double()
    r = torch.from_numpy(rows).cuda()
    pairs = (y[r] @ y.T) * (x[r] @ x.T)
    M = torch.stack([pairs[:, off[i]:off[i + 1]].sum(1) for i in range(B)], 1)
    want = (M ** 2).sum(0) / ((y[r] ** 2).sum(1) * (x[r] ** 2).sum(1)).sum()
    assert ((F2.double() - want).norm() / want.norm()).item() <= TOL
