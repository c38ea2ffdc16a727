"""The tridiagonal route of isopo_transform_spectral and the rule that leaves a K to the Jacobi kernel instead: matrices
whose reduction stops early (diagonal, block diagonal, repeated eigenvalues), sizes around the warp and row-block limits,
a negative or nearly null direction, and a batch in which only some layers need the second kernel.

Bounds: eigenvalues 2^-24 of their own size (float32 output of a float64 reduction) + 1e-12 of the largest on the first
route, 2e-6 of the largest on the second; coefficients 1e-5 + 1e-7 cond as everywhere in the spectral tests."""

import numpy as np
import pytest
import torch

from oracle import isopo_oracle as orc
from tests._util import rel_fro

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def b():
    from paper_2512_23353_b200 import binding
    return binding


def _with_spectrum(D, seed):
    Q, _ = np.linalg.qr(np.random.default_rng(seed).standard_normal((len(D), len(D))))
    K = (Q * D) @ Q.T
    return np.ascontiguousarray(((K + K.T) / 2).astype(np.float32))


def _run(b, Ks, A, lams, cutoff=0.0):
    B, n = len(A), len(Ks)
    info = torch.zeros(1, dtype=torch.int32, device="cuda")
    cs, es = ([torch.full((B,), float("nan"), device="cuda") for _ in range(n)] for _ in range(2))
    b.isopo_transform_spectral_batched([torch.from_numpy(K).cuda() for K in Ks], torch.from_numpy(A).cuda(), lams, cs, info,
                                       rel_cutoff=cutoff, eigenvalues=es)
    torch.cuda.synchronize()
    assert int(info.item()) == 0
    return [c.cpu().numpy() for c in cs], [e.cpu().numpy() for e in es]


def _check(K, A, lam, cutoff, c, e, values_tol):
    c_o, D_o = orc.spectral_coefficients(K.astype(np.float64), A.astype(np.float64), lam, cutoff)
    assert np.all(np.abs(e - D_o) <= values_tol(np.abs(D_o), D_o[0]))
    kept = D_o[D_o > cutoff * D_o[0]]
    cond = (kept[0] + lam) / (kept[-1] + lam)
    assert rel_fro(c, c_o) <= 1e-5 + 1e-7 * cond


FIRST = lambda d, top: 2.0 ** -24 * d + 1e-12 * top  # noqa: E731
SECOND = lambda d, top: 2e-6 * top  # noqa: E731


@pytest.mark.parametrize("B", [1, 2, 3, 4, 16, 32, 63, 64, 65, 128, 129, 130, 193, 255, 256])
@pytest.mark.parametrize("kind", ["spread", "repeated", "diagonal", "identity", "blocks"])
def test_first_route(b, B, kind):
    rng = np.random.default_rng(B)
    D = np.exp(rng.uniform(np.log(1e-3), np.log(30.0), size=B))
    if kind == "repeated":
        D = np.where(np.arange(B) % 2 == 0, 2.0, 0.5)
    K = _with_spectrum(D, B) if kind in ("spread", "repeated") else np.diag(D.astype(np.float32))
    if kind == "identity":
        K = 3.0 * np.eye(B, dtype=np.float32)
    if kind == "blocks":
        h = B // 2
        K = np.zeros((B, B), np.float32)
        K[:h, :h], K[h:, h:] = _with_spectrum(D[:h], 1) if h else 0.0, _with_spectrum(D[h:], 2)
    A = rng.standard_normal(B).astype(np.float32)
    lam = float(np.float32(0.01))
    cs, es = _run(b, [K], A, [lam])
    _check(K, A, lam, 0.0, cs[0], es[0], FIRST)


def test_scale_is_free(b):
    K = _with_spectrum(np.linspace(0.1, 3.0, 70), 3)
    A = np.random.default_rng(1).standard_normal(70).astype(np.float32)
    for scale in (np.float32(2.0 ** -60), np.float32(2.0 ** 60)):
        cs, es = _run(b, [K * scale], A, [float(scale) * 0.125])
        _check(K, A, 0.125, 0.0, cs[0] * scale, es[0] / scale, FIRST)


def test_layers_that_need_the_eigenvectors(b):
    """One well-conditioned layer, one with a negative eigenvalue (dropped), one whose small directions are cut off."""
    B = 48
    D = np.linspace(1.0, 4.0, B)
    neg, cut = D.copy(), D.copy()
    neg[0], cut[:5] = -0.5, 1e-3
    Ks = [_with_spectrum(d, 10 + i) for i, d in enumerate((D, neg, cut))]
    A = np.random.default_rng(2).standard_normal(B).astype(np.float32)
    lam = float(np.float32(0.05))
    cs, es = _run(b, Ks, A, [lam] * 3, 0.01)
    for K, c, e, tol in zip(Ks, cs, es, (FIRST, SECOND, SECOND)):
        _check(K, A, lam, 0.01, c, e, tol)
