"""GPU parity of the stand-alone weight gradient (Alg. 1: grad += advantages * rescaled gradient) where a tile of dW is summed by
one pair or CTA alone and written, not added to a cleared dW: few tokens, wide layers.

The coefficient is applied to the narrower operand in bf16 (or to the landed dY rows, one row of tiles), which the reference
repeats bit for bit; what is left is float32 sums of at most 512 exact products, 512 * 2^-24 = 3e-5 at the worst and some 1e-6 in
norm.  1e-5 is asked for."""

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu
TOL = 1e-5


@pytest.fixture(scope="module")
def b():
    from paper_2512_23353_b200 import binding
    return binding


def _case(Ls, d_in, d_out, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    off = np.concatenate([[0], np.cumsum(Ls)]).astype(np.int64)
    T = int(off[-1])
    X = torch.randn((T, d_in), device="cuda", generator=gen).bfloat16()
    dY = torch.randn((T, d_out), device="cuda", generator=gen).bfloat16()
    c = torch.randn(len(Ls), device="cuda", generator=gen)
    rows = c[torch.from_numpy(np.repeat(np.arange(len(Ls)), Ls)).cuda()][:, None]
    one_cta = ((d_out + 127) // 128) % 2 == 1 and (d_out + 127) // 128 < 7
    if one_cta or d_out <= d_in:
        want = (rows * dY.float()).bfloat16().double().T @ X.double()
    else:
        want = dY.double().T @ (rows * X.float()).bfloat16().double()
    return X, dY, c, off, want


def _run(b, X, dY, c, off, dW, beta):
    ws = b.alloc_workspace(b.BF16, X.shape[0], X.shape[1], dY.shape[1], len(off) - 1, b.PATH_GRAM)
    info = torch.zeros(1, dtype=torch.int32, device="cuda")
    b.isopo_weight_grad(X, dY, c, off, dW, ws, info, b.PATH_GRAM, beta)
    torch.cuda.synchronize()
    assert int(info.item()) == 0


@pytest.mark.parametrize("Ls,d_in,d_out", [
    ([1], 2304, 2560),                 # one token, more tiles than pairs
    ([3, 60, 1], 2056, 4104),          # one stage exactly; widths 8 past the tile grid
    ([20, 45], 4104, 2056),            # a second stage of one token
    ([5] * 100, 3072, 6144),           # eight stages, as many as writing a tile takes; more than 2^24 elements
    ([7] * 80, 3072, 6144),            # nine stages
    ([30, 30], 896, 256),              # two tiles of one stage
    ([33, 7, 1], 1000, 328),           # one row of CTAs, no pairs
    ([9] * 30, 200, 72),               # one CTA
])
@pytest.mark.parametrize("shift", [0, 4])  # dW at a 32-byte boundary, and 16 bytes behind one
def test_written_tiles(b, Ls, d_in, d_out, shift):
    X, dY, c, off, want = _case(Ls, d_in, d_out, 7 * d_in + d_out)
    raw = torch.full((d_out * d_in + 8,), float("nan"), device="cuda")
    dW = raw[shift:shift + d_out * d_in].view(d_out, d_in)
    _run(b, X, dY, c, off, dW, 0.0)
    assert ((dW.double() - want).norm() / want.norm()).item() <= TOL
    edge = torch.cat([raw[:shift], raw[shift + d_out * d_in:]])
    assert torch.isnan(edge).all()  # nothing beside dW is written
    dW.fill_(2.0)
    _run(b, X, dY, c, off, dW, 1.0)
    # 2 + dW rounded to float32 once more: up to 2^-24 of the sum's size per element
    assert ((dW.double() - 2.0 - want).norm() / want.norm()).item() <= TOL + 2.0 ** -24 * dW.double().norm().item() / want.norm().item()


@pytest.mark.parametrize("Ls,d_in,d_out", [
    ([111] * 60, 512, 600),      # five rows of tiles: just above a thousand stages of tiles (coefficient at the drain)
    ([50] * 140, 512, 600),      # the same through the scaled operand
    ([64] * 99, 512, 600),       # just below
    ([3, 5], 4104, 264),         # three rows, many columns of tiles
    ([1001] * 50, 512, 128),     # one row, two tiles
    ([4000] * 25, 64, 72),       # one tile
    ([15] * 1000, 4096, 104),    # one row of a wide layer
])
def test_few_rows_of_tiles(b, Ls, d_in, d_out):
    """Whole numbers small enough for every step of every kernel to be exact (a scaled operand of at most 8, float32 sums below 2^24): dW
    has to be what float64 gives, to the bit, whether the coefficient is applied to an operand or at the drain."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(d_in + len(Ls))
    off = np.concatenate([[0], np.cumsum(Ls)]).astype(np.int64)
    draw = lambda n, *shape: torch.randint(-n, n + 1, shape, device="cuda", generator=gen)  # noqa: E731
    X, dY, c = draw(1, int(off[-1]), d_in).bfloat16(), draw(1, int(off[-1]), d_out).bfloat16(), draw(8, len(Ls)).float()
    rows = c[torch.from_numpy(np.repeat(np.arange(len(Ls)), Ls)).cuda()][:, None]
    want = (rows.double() * dY.double()).T @ X.double()
    dW = torch.full((d_out, d_in), float("nan"), device="cuda")
    _run(b, X, dY, c, off, dW, 0.0)
    assert torch.equal(dW.double(), want)
    before = draw(1 << 12, d_out, d_in).float()
    dW.copy_(before)
    _run(b, X, dY, c, off, dW, 1.0)
    assert torch.equal(dW.double(), before.double() + want)
