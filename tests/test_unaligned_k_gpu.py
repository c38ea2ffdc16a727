"""K that starts at an odd element of a larger buffer (several K carved out of one allocation): every kernel that writes K, and
every kernel that reads it, takes a K that is 4-byte aligned and no more.

The transforms against the float64 oracle on the same float32 K, with the bounds of the aligned tests; the Gram kernels against
themselves on an aligned K, with room for another order of the float additions."""

import numpy as np
import pytest
import torch

from oracle import isopo_oracle as orc
from tests._util import VARIANT_NAME, rel_fro

pytestmark = pytest.mark.gpu

SIMPLE = [0, 1, 2, 3, 4, 6]
PQR = [-0.5, -0.5, 0.25, 0.01, 0.02, 0.03]


@pytest.fixture(scope="module")
def b():
    from paper_2512_23353_b200 import binding
    return binding


def _at_odd_element(a, shift=1):
    """The same values, `shift` elements into a buffer of their own (16-byte aligned by itself)."""
    flat = torch.empty(a.numel() + 4, device="cuda")
    view = flat[shift:shift + a.numel()].view(a.shape)
    view.copy_(a)
    assert flat.data_ptr() % 16 == 0 and view.data_ptr() % 16 == 4 * shift and view.is_contiguous()
    return view


def _problem(B, seed=0):
    rng = np.random.default_rng(1000 * seed + B)
    J = rng.standard_normal((B, 4 * B + 8)) / np.sqrt(4 * B)
    K = (J @ J.T).astype(np.float32)
    K = np.ascontiguousarray((K + K.T) / 2)
    A = rng.standard_normal(B).astype(np.float32)
    return K, A, float(np.float32(0.1 * np.mean(np.diag(K))))


def _want(K, A, v, lam):
    pqr, regs = (tuple(PQR[:3]), tuple(PQR[3:])) if v == 4 else (None, None)
    return orc.transform_advantages(K.astype(np.float64), A.astype(np.float64), VARIANT_NAME[v], lam, pqr, regs)


# multiples of four (rows that could be read 16 bytes at a time) on both sides of every kernel's range of sizes
@pytest.mark.parametrize("B", [4, 64, 128, 132, 256])
@pytest.mark.parametrize("shift", [1, 2, 3])
def test_transforms(b, B, shift):
    K, A, lam = _problem(B)
    Kd, Ad = _at_odd_element(torch.from_numpy(K).cuda(), shift), torch.from_numpy(A).cuda()
    info = torch.zeros(1, dtype=torch.int32, device="cuda")
    for v in SIMPLE + [5]:
        c, c2 = torch.empty(B, device="cuda"), [torch.empty(B, device="cuda") for _ in range(2)]
        pqr = PQR if v == 4 else None
        b.isopo_transform_advantages(Kd, Ad, v, lam, c, info, pqr)
        b.isopo_transform_advantages_batched([Kd, Kd], Ad, v, [lam, lam], c2, info, pqr)
        want = _want(K, A, v, lam)
        assert rel_fro(c.cpu().numpy(), want) <= 1e-5, v
        assert torch.equal(c, c2[0]) and torch.equal(c, c2[1])
    state = torch.zeros(4, device="cuda")
    b.isopo_reg_ema_update(Kd, 0.9, state)
    K64 = K.astype(np.float64)
    F2 = (K64 ** 2).sum(1) / np.trace(K64)
    assert rel_fro(state.cpu().numpy(), [F2.mean(), np.trace(K64) / B, (F2 / np.diag(K64)).mean(), 1.0]) <= 1e-6
    for v in (1, 5):
        c = torch.empty(B, device="cuda")
        b.isopo_transform_advantages_rel(Kd, Ad, v, 0.1, state, c, info)
        assert rel_fro(c.cpu().numpy(), _want(K, A, v, 0.1 * float(state[0 if v == 1 else 1]))) <= 1e-5
    c, eig = torch.empty(B, device="cuda"), torch.empty(B, device="cuda")
    b.isopo_transform_spectral(Kd, Ad, lam, c, info, eigenvalues=eig)
    assert rel_fro(c.cpu().numpy(), _want(K, A, 5, lam)) <= 1e-5
    assert rel_fro(eig.cpu().numpy(), np.linalg.eigvalsh(K64)[::-1]) <= 1e-5
    assert int(info.item()) == 0


@pytest.mark.parametrize("B", [128, 256, 260, 512])
def test_large_solve(b, B):
    K, A, lam = _problem(B, 1)
    ws = torch.empty(b.isopo_transform_large_workspace_bytes(B), dtype=torch.uint8, device="cuda")
    c, info = torch.empty(B, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")
    b.isopo_transform_advantages_large(_at_odd_element(torch.from_numpy(K).cuda()), torch.from_numpy(A).cuda(), lam, c, ws, info)
    torch.cuda.synchronize()
    assert int(info.item()) == 0 and rel_fro(c.cpu().numpy(), _want(K, A, 5, lam)) <= 1e-5


@pytest.mark.parametrize("dtype,path", [("f32", 1), ("f32", 2), ("bf16", 1), ("bf16", 2)])
@pytest.mark.parametrize("B", [8, 40])
def test_layer_gram_writes_it(b, dtype, path, B):
    code, dt = (b.F32, torch.float32) if dtype == "f32" else (b.BF16, torch.bfloat16)
    g = torch.Generator(device="cuda")
    g.manual_seed(B)
    T = 9 * B
    X, dY = (torch.empty(T, 64, device="cuda").normal_(generator=g).to(dt) for _ in range(2))
    off, info = np.arange(B + 1) * 9, torch.zeros(1, dtype=torch.int32, device="cuda")
    ws = b.alloc_workspace(code, T, 64, 64, B, path)
    K = torch.empty(B, B, device="cuda")
    odd = _at_odd_element(torch.full((B, B), float("nan"), device="cuda"))
    for out in (K, odd):
        b.isopo_layer_gram(X, dY, off, out, ws, info, path)
    torch.cuda.synchronize()
    assert int(info.item()) == 0 and torch.equal(odd, odd.T)
    # float32 additions of the same numbers in another order
    assert rel_fro(odd.cpu().numpy(), K.cpu().numpy()) <= 1e-6
