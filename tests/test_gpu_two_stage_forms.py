"""The forms that the two-stage reduction takes a batch in: what a layer gives must not depend on them."""
import numpy as np
import pytest

from paper_1806_04090_b200 import synth

pytestmark = pytest.mark.gpu


def _mat(m, n):
    return synth.lowrank_plus_noise(np.random.default_rng([92, m, n]), m, n, 1.0, noise_rel=0.5)


def _encode(a, layers, s=6.0, **kw):
    import torch
    from paper_1806_04090_b200 import api
    shapes = [tuple(t.shape) for t in layers]
    buf = torch.zeros(api.payload_bytes_spectral(shapes, 64), dtype=torch.uint8, device="cuda")
    return a.atomo_encode_spectral(layers, s, 17, step=3, k_cap=64, payload=buf, **kw)


@pytest.fixture(scope="module")
def atomo():
    from paper_1806_04090_b200 import api
    a = api.Atomo(0)
    yield a
    a.close()


# one layer of many on its own, on clusters of 256 columns per CTA, and in a batch of so many that they get 1024 columns per CTA
@pytest.mark.parametrize("m,n,few,many", [(600, 1210, 3, 40), (1025, 2050, 9, 20), (1500, 3004, 14, 16), (2049, 4100, 3, 9)])
def test_chase_on_clusters_of_either_size(atomo, m, n, few, many):
    import torch
    t = torch.from_numpy(_mat(m, n)).cuda()
    got = []
    for count in (1, few, many):
        pay, dbg = _encode(atomo, [t] * count, debug=True)
        hdrs = pay.headers()
        assert all(h.status == 0 for h in hdrs[1])
        got.append((dbg.layer_prob(0, m).copy(), pay.layer_arrays(0, hdrs)))
        for l in range(count):
            assert np.array_equal(dbg.layer_sigma(l, m), dbg.layer_sigma(0, m))
    sig = np.linalg.svd(_mat(m, n).astype(np.float64), compute_uv=False)
    for prob, arr in got:
        # (few layers' band reduction cuts its sums elsewhere than many's: fp32 runs of 32 products, 1e-8 of the largest eigenvalue,
        # over singular values of at least a hundredth of the largest)
        assert np.abs(prob - got[0][0]).max() <= 1e-7
        assert np.array_equal(arr["idx"], got[0][1]["idx"])
        short = arr["U"].astype(np.float64)
        norms = np.linalg.norm(_mat(m, n).T.astype(np.float64) @ short, axis=0)
        assert np.abs(norms - sig[arr["idx"]]).max() <= 1e-6 * sig[0]
