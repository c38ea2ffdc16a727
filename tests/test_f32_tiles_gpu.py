"""float32 kernels at the edges of their tiles: both tile sizes of the token GEMM, widths that are and are not multiples of
four (16-byte / 4-byte copies), row blocks of the K pass (16, 32, 64 sequences, several blocks, a padded last one), more
sequences than travel as kernel arguments, token tiles of the Gram and sampled kernels, both forms of the combine.

Bounds.  G is a float32 sum of L products (relative error about 2^-24 sqrt(L) and at most L 2^-24; L <= 300 here), K and
the combine add in float64: 2e-6 on K and dW.  Gram route: P and Q are float32 sums over the features, the rest float64.
The stand-alone weight gradient adds all T tokens in float32: 2e-6 too (T <= 2000)."""

import numpy as np
import pytest
import torch

from oracle import isopo_oracle as orc
from tests._util import rel_fro, to_f64

pytestmark = pytest.mark.gpu
TOL = 2e-6


@pytest.fixture(scope="module")
def b():
    from paper_2512_23353_b200 import binding
    return binding


def _problem(d_in, d_out, lens, seed):
    rng = np.random.default_rng(seed)
    off = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    to = lambda a: torch.from_numpy(a.astype(np.float32)).cuda()  # noqa: E731
    # a component common to all tokens gives K off-diagonals of its diagonal's size
    X = to(rng.standard_normal((off[-1], d_in)) + rng.standard_normal(d_in))
    dY = to(0.1 * (rng.standard_normal((off[-1], d_out)) + rng.standard_normal(d_out)))
    c = to(rng.standard_normal(len(lens)))
    return X, dY, off, c, orc.sequence_gradients(to_f64(X), to_f64(dY), off)


def _layer(b, X, dY, off, c, path):
    B = len(off) - 1
    ws = b.alloc_workspace(b.F32, int(off[-1]), X.shape[1], dY.shape[1], B, path)
    ws.fill_(0xFF)
    K, info = torch.empty(B, B, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")
    dW = torch.ones(dY.shape[1], X.shape[1], device="cuda")
    b.isopo_layer_gram(X, dY, off, K, ws, info, path)
    b.isopo_weight_grad(X, dY, c, off, dW, ws, info, path, 1.0)
    torch.cuda.synchronize()
    assert int(info.item()) == 0
    return K.cpu().numpy(), dW.cpu().numpy() - 1.0


SHAPES = [
    ([1, 17, 300, 16], 64, 64),
    ([5], 3, 1),
    ([40, 1, 15], 129, 67),                      # odd widths: 4-byte copies, padded gradients
    ([3 + i % 5 for i in range(16)], 132, 60),
    ([1 + i % 7 for i in range(17)], 100, 36),
    ([2 + i % 3 for i in range(33)], 256, 384),  # 128-wide tiles (198 CTAs stand-alone, 198 per-sequence)
    ([2 + i % 3 for i in range(64)], 255, 384),  # 128-wide tiles, odd width
    ([1 + i % 4 for i in range(65)], 68, 12),    # two row blocks, the second with one sequence
    ([1 + i % 3 for i in range(200)], 36, 20),
    ([1 + i % 2 for i in range(400)], 20, 12),   # offsets through device memory
    ([2, 5], 900, 640),                          # combine whole (over 2^19 elements)
    ([300, 299, 301, 633], 40, 21),              # Gram tiles of 64 (300 of them), the last one ragged
]


@pytest.mark.parametrize("case", range(len(SHAPES)))
@pytest.mark.parametrize("route", ["gram", "stored"])
def test_layer(b, case, route):
    lens, d_in, d_out = SHAPES[case]
    X, dY, off, c, G = _problem(d_in, d_out, lens, case)
    K, dW = _layer(b, X, dY, off, c, b.PATH_GRAM if route == "gram" else b.PATH_MATERIALISE)
    want = orc.weight_gradient(G, to_f64(c))
    assert rel_fro(K, orc.ntk(G)) <= TOL
    assert np.array_equal(K, K.T)
    # dW is read back around a base of one: its float32 rounding there
    assert rel_fro(dW, want) <= TOL + 1.2e-7 * np.sqrt(want.size) / np.linalg.norm(want)


@pytest.mark.parametrize("n_samples", [1, 63, 65, 130])
@pytest.mark.parametrize("d_in,d_out", [(64, 48), (37, 130)])
@pytest.mark.parametrize("lens", [[1, 70, 64, 33, 129], [4000, 5000, 600, 1]])  # tiles of 32; of 64 for 65 and 130 samples
def test_sampled(b, n_samples, d_in, d_out, lens):
    X, dY, off, A, G = _problem(d_in, d_out, lens, n_samples + d_in)
    B, T = len(off) - 1, int(off[-1])
    rows = np.random.default_rng(n_samples).permutation(T)[:n_samples].astype(np.int64)
    ws = b.alloc_sampled_workspace(b.F32, T, d_in, d_out, B, n_samples)
    cc, F2, info = torch.empty(B, device="cuda"), torch.empty(B, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")
    b.isopo_sampled_coefficients(X, dY, off, rows, A, 0.0, cc, ws, info, F2)
    torch.cuda.synchronize()
    want, _, _ = orc.isopo_layer_sampled(to_f64(X), to_f64(dY), off, to_f64(A), rows, 0.0)
    assert int(info.item()) == 0
    assert rel_fro(F2.cpu().numpy(), want) <= 2 * TOL  # a square


@pytest.mark.parametrize("T", [1, 15, 16, 17, 127, 128, 129, 300, 2049])
@pytest.mark.parametrize("d_in,d_out", [(8, 8), (64, 65), (520, 260), (2048, 1280)])
def test_weight_gradient_slabs(T, d_in, d_out):
    """The GEMM over all tokens cuts them into as many slabs as make its waves cheapest: one, or down to 16 tokens; few tiles and
    many.  Bound: float32 products and sums over at most T terms and the slabs' float32 additions, T 2^-24 at worst, taken as 2e-6
    of the norm (random signs)."""
    from paper_2512_23353_b200 import binding as b
    B = min(T, 3)
    off = np.linspace(0, T, B + 1).astype(np.int64)
    g = torch.Generator(device="cuda").manual_seed(T + d_in)
    X, dY = torch.randn(T, d_in, device="cuda", generator=g), torch.randn(T, d_out, device="cuda", generator=g)
    c, dW = torch.randn(B, device="cuda", generator=g), torch.full((d_out, d_in), float("nan"), device="cuda")
    info = torch.zeros(1, dtype=torch.int32, device="cuda")
    ws = b.alloc_workspace(b.F32, T, d_in, d_out, B, b.PATH_GRAM)
    per_token = c.double().repeat_interleave(torch.from_numpy(np.diff(off)).cuda())[:, None]
    want = (per_token * dY.double()).T @ X.double()
    for beta in (0.0, 1.0):
        b.isopo_weight_grad(X, dY, c, off, dW, ws, info, b.PATH_GRAM, beta)
        assert float((dW.double() - (1 + beta) * want).norm() / want.norm()) <= 2e-6 * (1 + beta)
    assert int(info.item()) == 0
