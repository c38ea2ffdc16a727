"""float32 stand-alone weight gradient where the choice of tiles and token slabs changes: slabs for one CTA of 128 x 128 to an SM, for two,
one slab of few tokens, 64 x 64; against torch float64.  A dW entry is a float32 sum over T tokens (a fraction of 2^-24 sqrt(T) of its
norm at random signs, far below for sums that meet across slabs): 2e-6, as for the other float32 kernels."""

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Ls,d_in,d_out", [([100] * 5, 896, 896), ([2000] * 10, 128, 128), ([20], 1536, 1536), ([50] * 4, 1152, 1151), ([140, 140], 1536, 1539),
                                           ([250] * 10, 379, 635), ([1] * 3, 2000, 1999), ([311] * 16, 1024, 80), ([500] * 4, 513, 512)])
@pytest.mark.parametrize("beta", [0.0, 1.0])
def test_weight_grad(Ls, d_in, d_out, beta):
    from paper_2512_23353_b200 import binding as b
    off, B, T = np.concatenate([[0], np.cumsum(Ls)]).astype(np.int64), len(Ls), sum(Ls)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(T + d_in)
    X, dY, c = (torch.randn(s, device="cuda", generator=gen) for s in ((T, d_in), (T, d_out), (B,)))
    dW = torch.randn((d_out, d_in), device="cuda", generator=gen) if beta else torch.full((d_out, d_in), float("nan"), device="cuda")
    want = (dY.double() * c.double()[torch.from_numpy(np.repeat(np.arange(B), Ls)).cuda(), None]).T @ X.double()
    if beta:
        want += dW.double()
    info = torch.zeros(1, dtype=torch.int32, device="cuda")
    b.isopo_weight_grad(X, dY, c, off, dW, b.alloc_workspace(b.F32, T, d_in, d_out, B, b.PATH_GRAM), info, b.PATH_GRAM, beta)
    torch.cuda.synchronize()
    assert int(info.item()) == 0
    assert ((dW.double() - want).norm() / want.norm()).item() <= 2e-6
