"""Singular values of every atom: both forms of the eigenvalue kernel (two and four lanes per eigenvalue) at the edges of its
CTAs, on spectra that its brackets find hard."""
import numpy as np
import pytest
import torch

from paper_1806_04090_b200 import api

pytestmark = pytest.mark.gpu

MANY = 16384                                     # eigenvalues in a call from which two lanes take one


def _matrix(r, kind):
    rng = np.random.default_rng(r)
    q = np.linalg.qr(rng.standard_normal((r, r)))[0]
    if kind == "flat":
        return rng.standard_normal((r, r + 7)).astype(np.float32)
    if kind == "pairs":                          # neighbouring values agree to a few last digits
        sv = np.repeat(np.linspace(1.0, 2.0, (r + 1) // 2), 2)[:r] * (1.0 + 1e-7 * (np.arange(r) % 2))
    elif kind == "graded":
        sv = 2.0 ** -np.linspace(0.0, 10.0, r)
    else:                                        # "rank": a few values, the others zero
        sv = np.where(np.arange(r) < max(1, r // 8), 1.0 + np.arange(r), 0.0)
    return (q * sv @ np.linalg.qr(rng.standard_normal((r, r)))[0].T).astype(np.float32)


@pytest.mark.parametrize("kind", ["flat", "pairs", "graded", "rank"])
def test_both_forms_against_svd(kind):
    sizes = [1, 2, 3, 8, 9, 15, 16, 17, 31, 32, 33, 63, 64, 65, 130]
    mats = [_matrix(r, kind) for r in sizes]
    dev = [torch.from_numpy(m).cuda() for m in mats]
    fill = torch.randn(64, 80, device="cuda")
    few = dev
    many = dev + [fill] * (MANY // 64 + 1)
    assert sum(min(m.shape) for m in few) < MANY <= sum(min(m.shape) for m in many)
    a = api.Atomo(0)
    got = []
    for layers in (few, many):
        pay, dbg = a.atomo_encode_spectral(layers, 1.0, seed=1, step=0, k_cap=16, debug=True)
        assert all(h.status == 0 for h in pay.headers()[1])
        got.append([dbg.layer_sigma(i, r).astype(np.float64) for i, r in enumerate(sizes)])
    for r, m, x, y in zip(sizes, mats, *got):
        exact = np.linalg.svd(m.astype(np.float64), compute_uv=False)
        lam = exact[0] ** 2
        # the fp32 Gram matrix is off by at most sqrt(r) roundings of its entries, its eigenvalues by no more
        bar = 4.0 * np.sqrt(r) * 2.0 ** -24 * lam
        assert np.abs(x ** 2 - exact ** 2).max() <= bar, (kind, r)
        # the forms agree to the final bracket (4e-13 of an extent of at most 3 lam) and the rounding of lambda and sigma to fp32
        assert np.all(np.abs(x ** 2 - y ** 2) <= 2.0 ** -21 * x ** 2 + 2e-12 * lam), (kind, r)
    a.close()
