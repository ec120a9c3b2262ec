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


def test_routes_where_the_gpu_cannot_place_the_two_stage_reduction():
    """No room for the band reduction or for the chase's clusters: the batch takes the Jacobi routes, as if they had been asked for,
    and not an error.  Little room: the same kernels on fewer CTAs, or the chase's larger CTAs."""
    import torch
    from paper_1806_04090_b200 import api
    a, b = api.Atomo(0), api.Atomo(0)
    layers = [torch.from_numpy(_mat(m, n)).cuda() for m, n in ((40, 90), (1100, 1300), (600, 700))]
    small = layers[::2]                                             # no cluster of the chase is needed up to 1024 rows

    def run(ctx, what):
        pay, _ = _encode(ctx, what)
        return pay.buf.clone(), ctx.last_eig_scheme(), [h.status for h in pay.headers()[1]]

    b.set_persistent_eig(2)
    jacobi, jacobi_small = run(b, layers), run(b, small)
    b.set_persistent_eig(3)
    assert jacobi[1] < 3 and jacobi[2] == [0, 0, 0]
    full, full_small = run(b, layers), run(b, small)
    assert full[1] == 3 and full[2] == [0, 0, 0]
    for band, chase, want, want_small in ((0, -1, jacobi, jacobi_small), (-1, 0, jacobi, full_small), (7, -1, full, full_small),
                                          (-1, 1, full, full_small), (1, 1, full, full_small), (-1, -1, full, full_small)):
        a.limit_tridiag_route(band, chase)
        for what, expect in ((layers, want), (small, want_small)):
            got = run(a, what)
            assert got[1] == expect[1] and got[2] == [0] * len(what), (band, chase)
            assert torch.equal(got[0], expect[0]), (band, chase)
    a.limit_tridiag_route(5, -1)                                    # more CTAs per layer asked for than there is room
    a.set_tridiag_ctas(16)
    got = run(a, layers)
    assert got[1] == 3 and torch.equal(got[0], full[0])
    for bad in ((-2, 0), (0, -2)):
        with pytest.raises(api.AtomoError):
            a.limit_tridiag_route(*bad)
    a.close()
    b.close()
