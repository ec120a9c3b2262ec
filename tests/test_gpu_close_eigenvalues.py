"""Layers with equal or nearly equal singular values, many of them kept: the kept vectors must be an orthonormal set of eigenvectors, and
where all atoms are kept the payload must decode to the layer itself."""
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


def _layer(kind, r, n, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    rnd = lambda *s: torch.randn(*s, device="cuda", generator=gen)
    i, j = torch.arange(r, device="cuda"), torch.arange(n, device="cuda")
    if kind == "walsh":                                   # rows of +-1, orthogonal but for the last columns
        b = i[:, None] & j[None, :]
        for s in (16, 8, 4, 2, 1):
            b = b ^ (b >> s)
        return 1.0 - 2.0 * (b & 1).float()
    if kind == "identity":
        return torch.eye(r, n, device="cuda") * 2.0
    if kind == "constant":
        return torch.full((r, n), 0.37, device="cuda")
    if kind == "twice":                                   # two equal blocks: every singular value twice
        return torch.block_diag(*[rnd(r // 2, n // 2)] * 2)
    if kind == "equal rows":
        return rnd(r, n)[torch.randint(0, max(1, r // 3), (r,), device="cuda", generator=gen)]
    if kind == "row scales":
        return rnd(r, n) * torch.exp2(torch.randint(-20, 20, (r, 1), device="cuda", generator=gen).float())
    if kind == "graded":
        return rnd(r, n) * torch.logspace(0, -12, r, device="cuda")[:, None]
    if kind == "zero rows":
        return rnd(r, n) * (torch.rand(r, 1, device="cuda", generator=gen) < 0.4)
    assert kind == "low rank"
    return rnd(r, 5) @ rnd(5, n)


def _check(atomo, G, s, k_cap):
    tall = G.shape[0] > G.shape[1]
    pay, _ = atomo.atomo_encode_spectral([G], s, 5, step=3, k_cap=k_cap)
    hdrs = pay.headers()
    head = hdrs[1][0]
    assert head.status == 0 and head.k > 0
    arrays = pay.layer_arrays(0, hdrs)
    U = torch.from_numpy(arrays["V" if tall else "U"].astype(np.float64)).cuda()
    A = G.double().T @ G.double() if tall else G.double() @ G.double().T
    AU = A @ U
    # A is rounded to fp32 once (2^-24 of its norm), and so are the vectors; the reduction adds about as much again, and up to 512 rows every
    # eight reflectors of the back-transformation round the vector once more
    res = (AU - U * (U * AU).sum(0)).norm(dim=0) / torch.linalg.matrix_norm(A)
    r = U.shape[0]
    assert float(res.max()) <= (4.0 + (r / 8.0 if r <= 512 else 0.0)) * 2.0 ** -24, float(res.max())
    off = (U.T @ U - torch.eye(head.k, device="cuda")).abs()
    assert float(off.max()) <= 2e-6, float(off.max())
    return pay, head, off


@pytest.mark.parametrize("m,n", [(8, 1011), (17, 1694), (20, 1283), (39, 192), (57, 730), (64, 64), (96, 130), (130, 60), (352, 10)])
@pytest.mark.parametrize("kind", ["walsh", "identity", "constant", "twice", "equal rows", "row scales", "graded", "zero rows", "low rank"])
def test_all_atoms_kept(atomo, kind, m, n):
    r = min(m, n)
    if kind == "twice" and (m % 2 or n % 2):
        n, m = n + n % 2, m + m % 2
        r = min(m, n)
    for seed in range(3):
        G = _layer(kind, r, max(m, n), seed)
        if m > n:
            G = G.T.contiguous()
        if not float(G.abs().max()):
            continue
        pay, head, off = _check(atomo, G, float(2 * r), r)
        out = atomo.atomo_decode(pay)[0]
        # sum of u u^T G over an orthonormal basis (but for atoms whose singular value came out as zero: below sqrt(2^-24) of the largest, and then
        # at rounding level of the squares)
        assert float((out - G).norm()) <= (2.0 * float(off.norm()) + 2.0 ** -20) * float(G.norm())


# the vector kernels' instances above 512 rows, some atoms of each layer
@pytest.mark.parametrize("m,n,s", [(600, 900, 30.0), (1024, 1056, 40.0), (1100, 1300, 12.0), (2048, 2080, 60.0), (2100, 2304, 12.0)])
@pytest.mark.parametrize("kind", ["walsh", "identity", "twice", "constant", "equal rows"])
def test_large_layers(atomo, kind, m, n, s):
    _check(atomo, _layer(kind, m, n, 1), s, 128)
