"""Vectors of short sides of 1025 to 2048: one atom per CTA, or two at once on twice the warps, by the budget and the number of layers."""
import numpy as np
import pytest
import torch

from paper_1806_04090_b200 import api

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def atomo():
    a = api.Atomo(0)
    yield a
    a.close()


def _check_vectors(atomo, m, n, count, s, seed, step):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(m + count)
    G = torch.randn(m, n, device="cuda", generator=gen)
    pay, _ = atomo.atomo_encode_spectral([G] * count, s, seed, step=step, k_cap=128)
    hdrs = pay.headers()
    A = G.double() @ G.double().T
    top = float(torch.linalg.eigvalsh(A)[-1])
    seen = 0
    for l in range(count):
        k = hdrs[1][l].k
        assert hdrs[1][l].status == 0
        if not k:
            continue
        seen += k
        U = torch.from_numpy(pay.layer_arrays(l, hdrs)["U"].astype(np.float64)).cuda()
        AU = A @ U
        res = (AU - U * ((U * AU).sum(0) / (U * U).sum(0))).norm(dim=0) / top
        # every panel of the reduction rounds A's entries once, by at most 2^-25 of them and with either sign: sqrt(r / 8) of these in
        # all, over a column of A, whose norm (about 1.4 / r of the trace) is at most half of the largest eigenvalue (3.7 / r or more)
        assert float(res.square().mean().sqrt()) <= 2.0 ** -25 * np.sqrt(m / 8.0) * 0.5
        dots = U.T @ U
        assert float((dots - torch.eye(k, device="cuda")).abs().max()) <= 4e-7
    assert seen > 0
    return [h.k for h in hdrs[1]]


# one CTA per atom and to spare; several atoms per CTA from the start
@pytest.mark.parametrize("m,n,count,s", [(1025, 1030, 1, 5.0), (2047, 2048, 1, 8.0), (1100, 1200, 9, 3.0), (1100, 1200, 40, 6.0), (2048, 2060, 1, 60.0)])
def test_vectors_of_either_form(atomo, m, n, count, s):
    _check_vectors(atomo, m, n, count, s, 6, 1)


# a CTA per atom is expected (16 per layer for a budget of 9), and some layer keeps more atoms than that
@pytest.mark.parametrize("m,n,step", [(1100, 1200, 26), (1601, 1700, 19)])
def test_more_atoms_than_were_expected(atomo, m, n, step):
    kept = _check_vectors(atomo, m, n, 9, 9.0, 6, step)
    assert max(kept) > 16, kept
