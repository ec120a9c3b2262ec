"""Layers whose rows have entries far above the others: the integer Gram kernel must be as close to 64 bits as the fp32 FMA kernel."""
import numpy as np
import pytest
import torch

from paper_1806_04090_b200 import api

pytestmark = pytest.mark.gpu


def _layer(kind, r, n, gen):
    dev = torch.device("cuda")
    g = torch.randn(r, n, device=dev, generator=gen)
    rows = torch.arange(r, device=dev)
    if kind == "laplace":
        u = torch.rand(r, n, device=dev, generator=gen) - 0.5
        return torch.log1p(u.abs() * -2.0).clamp(min=-30.0) * -u.sign()
    if kind.startswith("t"):                         # Student's t with that many degrees of freedom
        dof = int(kind[1:])
        chi = sum(torch.randn(r, n, device=dev, generator=gen) ** 2 for _ in range(dof))
        return g / (chi / dof).sqrt()
    if kind.startswith("one"):                       # one entry of that size per row
        g[rows, torch.randint(0, n, (r,), device=dev, generator=gen)] = float(kind[3:])
    if kind.startswith("some"):                      # in every 50th row only: the others' tiles must not suffer
        g[rows[::50], torch.randint(0, n, (len(rows[::50]),), device=dev, generator=gen)] = float(kind[4:])
    if kind == "columns":                            # a few columns outweigh the rest
        g[:, :20] *= 100.0
    if kind == "sparse":
        g *= torch.rand(r, n, device=dev, generator=gen) < 0.02
    return g


def _errors(a, G, A, lam, V):
    r = min(G.shape)
    pay, dbg = a.atomo_encode_spectral([G], 48.0, seed=3, step=0, k_cap=128, debug=True)
    hdrs = pay.headers()
    assert hdrs[1][0].status == 0 and hdrs[1][0].k >= 16
    sigma = torch.from_numpy(dbg.layer_sigma(0, r).astype(np.float64)).to(lam)
    arrays = pay.layer_arrays(0, hdrs)
    U = torch.from_numpy(arrays["U" if G.shape[0] <= G.shape[1] else "V"].astype(np.float64)).to(lam)
    U = U / U.norm(dim=0)
    W = V[:, torch.from_numpy(arrays["idx"].astype(np.int64)).to(lam.device)]
    angle = (U - W * (U * W).sum(0)).norm(dim=0)
    AU = A @ U
    residual = (AU - U * (U * AU).sum(0)).norm(dim=0) / lam[0]
    return {"lambda": float((sigma ** 2 - lam).norm() / lam.norm()), "angle": float(angle.median()), "residual": float(residual.square().mean().sqrt())}


@pytest.mark.parametrize("m,n", [(600, 1101), (1101, 600), (1030, 4100)])
@pytest.mark.parametrize("kind", ["normal", "laplace", "t3", "t2", "t1", "one10", "one30", "one100", "one1000", "one1e4", "one1e6", "some30", "some1e6",
                                  "columns", "sparse"])
def test_no_further_from_64_bits_than_the_fma_kernel(kind, m, n):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(m + 3 * n)
    G = _layer(kind, min(m, n), max(m, n), gen)
    A = G.double() @ G.double().T
    lam, V = torch.linalg.eigh(A)
    lam, V = lam.flip(0), V.flip(1)
    if m > n:
        G = G.T.contiguous()
    a = api.Atomo(0)
    got = _errors(a, G, A, lam, V)
    a.set_gram_path(0)
    fma = _errors(a, G, A, lam, V)
    a.close()
    print(kind, m, n, " ".join("%s %.2e | %.2e" % (k, got[k], fma[k]) for k in got))
    # both carry the reduction's own rounding (3e-8 of the largest eigenvalue and less) and differ from seed to seed by some
    # tens of per cent; what the left-out digit pairs did to such rows was a factor of two to five
    for k, extra in (("lambda", 2e-9), ("angle", 0.0), ("residual", 2e-9)):
        assert got[k] <= 1.3 * fma[k] + extra, (k, got, fma)
