"""Room for the integer digits of the Gram matrices: shared by the layers of a call, and done without where there is none."""
import numpy as np
import pytest
import torch

from paper_1806_04090_b200 import api

pytestmark = pytest.mark.gpu


def _layer(m, n, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    return torch.randn(m, n, device="cuda", generator=gen)


def _sigma(a, G):
    pay, dbg = a.atomo_encode_spectral(G, 2.0, seed=3, step=0, k_cap=32, debug=True)
    assert all(h.status == 0 for h in pay.headers()[1])
    return [dbg.layer_sigma(l, min(g.shape)).copy() for l, g in enumerate(G)]


def test_layers_in_several_groups():
    G = [_layer(1030, 9001, l) for l in range(30)]              # 1.1 GB of digits: two groups, rows of two passes
    G[3] = _layer(1100, 1300, 3)
    a = api.Atomo(0)
    many = _sigma(a, G)
    for l in (0, 3, 27, 28, 29):
        one = _sigma(a, [G[l]])[0]
        assert np.array_equal(many[l], one)                     # integer sums: the company does not show
        lam = torch.linalg.eigvalsh(G[l].double() @ G[l].double().T).flip(0).cpu().numpy()
        assert np.abs(one.astype(np.float64) ** 2 - lam).max() <= 4.0 * 2.0 ** -24 * np.linalg.norm(lam)
    a.close()


@pytest.mark.parametrize("m,n", [(1100, 1301), (300, 40001)])
def test_no_room_for_digits(m, n):
    G = [_layer(m, n, 5)]
    a = api.Atomo(0)
    with_digits = _sigma(a, G)[0]
    a.set_gram_path(0)
    without = _sigma(a, G)[0]
    a.close()
    assert not np.array_equal(with_digits, without)
    lo, hi = 0, 1 << 30                                         # the least workspace that will do, to 64 KB
    while hi - lo > 1 << 16:
        mid = (lo + hi) // 2
        b = api.Atomo(0)
        b.limit_workspace(mid)
        try:
            got = _sigma(b, G)[0]
            hi = mid
        except api.AtomoError as e:
            assert api.STATUS_NAMES[e.code] == "CUDA"
            lo = mid
            b.limit_workspace(-1)
            assert np.array_equal(_sigma(b, G)[0], with_digits)  # the context works on
        b.close()
    b = api.Atomo(0)
    b.limit_workspace(hi)
    for _ in range(2):
        assert np.array_equal(_sigma(b, G)[0], without)
    b.limit_workspace(hi + 4 * m * (n + 64) + 148 * 128 * 128 * 8 + (1 << 20))   # the digits, and a partial tile in fp64 per SM
    assert np.array_equal(_sigma(b, G)[0], with_digits)
    with pytest.raises(api.AtomoError):
        b.limit_workspace(-2)
    b.close()
