"""The integer Gram kernel at the edges of its tiles, digits and parts: singular values against 64 bits."""
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


def _sigma(a, G):
    r = min(G.shape)
    pay, dbg = a.atomo_encode_spectral([G], 2.0, seed=3, step=0, k_cap=32, debug=True)
    return pay.headers()[1][0].status, dbg.layer_sigma(0, r).astype(np.float64)


def _check(a, G):
    status, s = _sigma(a, G)
    assert status == 0
    lam = torch.linalg.svdvals(G.double()).cpu().numpy() ** 2
    # rounding A's entries to fp32 moves an eigenvalue by at most 2^-24 ||A||_F; the reduction and the digits by as much again, each
    assert np.abs(s ** 2 - lam).max() <= 4.0 * 2.0 ** -24 * np.linalg.norm(lam)
    # the nuclear norm: a shift of all eigenvalues would show here (4e-9 of their mean is a fifth of what the digit pairs left out lack)
    assert abs((s ** 2).sum() - lam.sum()) <= 2.0 ** -23 * lam.sum()


@pytest.mark.parametrize("m,n", [(513, 517), (640, 641), (1025, 1026), (1152, 1153), (1153, 2049), (1025, 8191), (1025, 8193),   # rows, two passes
                                 (700, 513), (1100, 1037), (3001, 641), (1153, 1025),                                        # columns
                                 (17, 193), (129, 2049), (2047, 255), (16384, 18), (300, 65535),                             # narrow ones
                                 (520, 33001)])                                                                              # more columns than an accumulator holds
def test_edges(atomo, m, n):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(m * 7 + n)
    _check(atomo, torch.randn(m, n, device="cuda", generator=gen))


@pytest.mark.parametrize("n", [131072, 150001])
def test_parts_whose_sum_outgrows_53_bits(atomo, n):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(n)
    G = torch.randn(514, n, device="cuda", generator=gen)
    G[:, : n // 2] *= 0.001
    G[3] = G[2]                                                     # sums as large as the diagonal's off it
    status, s = _sigma(atomo, torch.empty(514, n + 1, device="cuda")[:, 1:].copy_(G))
    assert status == 0
    lam = torch.linalg.eigvalsh(G.double() @ G.double().T).flip(0).cpu().numpy()
    assert np.abs(s ** 2 - lam).max() <= 4.0 * 2.0 ** -24 * np.linalg.norm(lam)


def test_leading_dimension_and_scales(atomo):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(1)
    wide = torch.randn(1030, 2003, device="cuda", generator=gen)
    _check(atomo, wide[:, 1:1901])                                  # rows 4 bytes off, a pitch of 2003
    _check(atomo, wide[:, :1900] * 1e-15)
    rows = torch.exp2(torch.randint(-12, 12, (1030, 1), device="cuda", generator=gen).float())
    _check(atomo, (wide * rows).contiguous())                       # every vector has a unit of its own
    wide[7] = 0.0
    wide[3, 5] = 3.0e4                                              # one entry outweighs its vector (how close such rows come: test_gpu_gram_range.py)
    _check(atomo, wide)


def test_many_layers_of_middle_size_agree_with_one(atomo):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(2)
    G = [torch.randn(520, 4096, device="cuda", generator=gen) for _ in range(33)]     # above the number of elements that sends them here
    r = 520
    pay, dbg = atomo.atomo_encode_spectral(G, 2.0, seed=3, step=0, k_cap=32, debug=True)
    assert all(h.status == 0 for h in pay.headers()[1])
    for l in (0, 32):
        s = dbg.layer_sigma(l, r).astype(np.float64)
        lam = torch.linalg.svdvals(G[l].double()).cpu().numpy() ** 2
        assert np.abs(s ** 2 - lam).max() <= 4.0 * 2.0 ** -24 * np.linalg.norm(lam)


@pytest.mark.parametrize("bad", [float("inf"), float("-inf"), float("nan")])
@pytest.mark.parametrize("m,n", [(1030, 1100), (1100, 1030), (1030, 9001)])
def test_non_finite_entries(atomo, m, n, bad):
    G = torch.randn(m, n, device="cuda")
    G[m - 1, n - 1] = bad
    pay, _ = atomo.atomo_encode_spectral([G], 2.0, seed=3, step=0, k_cap=32)
    head = pay.headers()[1][0]
    assert head.status != 0 and head.k == 0
