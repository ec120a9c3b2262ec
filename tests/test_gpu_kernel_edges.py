"""The kernels at the sizes where their tiles, chunks and launch forms change: short sides around the forms of the two-stage
reduction and its chase, K ranges cut into parts, thread layouts of the spectral decode, more payloads, atoms, layers and
vectors than one round holds."""
import numpy as np
import pytest

from paper_1806_04090_b200 import synth
from tests import parity

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def atomo():
    import torch
    from paper_1806_04090_b200 import api
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    a = api.Atomo(0)
    yield a
    a.close()


def _mat(m, n):
    return synth.lowrank_plus_noise(np.random.default_rng([91, m, n]), m, n, 1.0, noise_rel=0.05)


# the same matrix `count` times: 1 = a cluster of 256 columns per CTA, more = as few CTAs per layer as hold it
@pytest.mark.parametrize("m,n,count", [(1024, 1030, 1), (1025, 1040, 1), (2048, 2052, 1), (2049, 2060, 1), (520, 530, 40),
                                       (1024, 1028, 20), (1100, 1110, 10), (2049, 2060, 5),
                                       # K range of the Gram matrix in parts: tall, or rows off the 16-byte grid
                                       (513, 18, 1), (16384, 17, 1), (4097, 256, 1), (4097, 257, 1), (65, 2049, 1), (300, 511, 2)])
def test_probabilities_and_vectors_against_svd(atomo, m, n, count):
    import torch
    G = _mat(m, n)
    t = torch.from_numpy(G).cuda()
    s = 3.0
    pay, dbg = atomo.atomo_encode_spectral([t] * count, s, 17, step=3, k_cap=64, debug=True)
    sig = np.linalg.svd(G.astype(np.float64), compute_uv=False)
    hdrs = pay.headers()
    r = min(m, n)
    want, left, budget = np.ones(r), float(sig.sum()), s            # Algorithm 1
    for i in range(r):
        if sig[i] * budget <= left:
            want[i:] = sig[i:] * budget / left
            break
        left, budget = left - sig[i], budget - 1.0
    for l in range(count):
        assert hdrs[1][l].status == 0
        # (nearly square noise: what the fp32 entries of the Gram matrix leave of the smallest singular values)
        assert np.abs(dbg.layer_prob(l, r) - want).max() <= (4e-6 if r > 512 else 2e-7)
        arr = pay.layer_arrays(l, hdrs)
        if arr["k"]:
            U, V = arr["U"].astype(np.float64), arr["V"].astype(np.float64)
            short = U if m <= n else V
            assert np.abs(short.T @ short - np.eye(arr["k"])).max() <= 2e-5
            got = np.linalg.norm((G.T if m <= n else G).astype(np.float64) @ short, axis=0)
            assert np.abs(got - sig[arr["idx"]]).max() <= 2e-5 * sig[0]


@pytest.mark.parametrize("m,n", [(1, 1), (17, 1), (5, 31), (129, 33), (64, 128), (70, 129), (100, 1024), (65, 1025), (33, 4100), (40, 4097)])
def test_decode_layouts(atomo, m, n):
    import torch
    G = _mat(m, n)
    t = torch.from_numpy(G).cuda()
    pay, _ = atomo.atomo_encode_spectral([t], 36.0, 3, step=1, k_cap=64)    # more than 32 atoms where there are as many
    hdrs = pay.headers()
    arr = pay.layer_arrays(0, hdrs)
    out = torch.full((m, n), float("nan"), device="cuda")
    atomo.atomo_decode(pay, out=[out])
    want = (arr["U"].astype(np.float64) * arr["coef"].astype(np.float64)) @ arr["V"].astype(np.float64).T
    assert np.abs(out.cpu().numpy() - want).max() <= 2e-6 * max(1e-30, np.abs(want).max()) * max(1, arr["k"])


def test_decode_many_layers_and_payloads(atomo):
    import torch
    from paper_1806_04090_b200 import api
    mats = [_mat(9 + l % 5, 12 + l % 3) for l in range(150)]
    ts = [torch.from_numpy(G).cuda() for G in mats]
    singles, pays = [], []
    for worker in range(35):
        buf = torch.empty(api.payload_bytes_spectral([G.shape for G in mats], 16), dtype=torch.uint8, device="cuda")
        pay, _ = atomo.atomo_encode_spectral(ts, 2.0, seed=50 + worker, step=2, k_cap=16, payload=buf)
        pays.append(pay)
        singles.append([o.double() for o in atomo.atomo_decode(pay)])
    avg = atomo.atomo_decode_average(pays)
    for l in range(len(mats)):
        want = sum(x[l] for x in singles) / len(pays)
        assert float((avg[l].double() - want).abs().max()) <= 2e-6 * float(want.abs().max()) + 1e-12


@pytest.mark.parametrize("compact", [False, True])
def test_more_vectors_than_a_launch_holds(compact):
    """27 vectors of one element to several chunks in one call: the decode of each equals the decode of a call of its own."""
    import torch
    from paper_1806_04090_b200 import api
    a = api.Atomo(0)
    if compact:
        a.set_entrywise_format(api.EW_COMPACT, sat_cap=1 << 12)
    rng = np.random.default_rng(8)
    lengths = ([1, 5, 4095, 4096, 4097, 70000, 1_000_003, 300_001, 12] * 3)[:27]
    gs = [torch.from_numpy(rng.laplace(size=n).astype(np.float32)).cuda() for n in lengths]
    for form in (0, 1, 2):
        a.set_entrywise_launch(form)
        pay, _ = a.atomo_encode_entrywise(gs, 500.0, seed=4, step=6, k_cap=4096)
        outs = [o.clone() for o in a.atomo_decode(pay)]
        hdrs = pay.headers()
        if form == 0:
            first, ks = outs, [h.k for h in hdrs[1]]
        assert all(h.status == 0 for h in hdrs[1]) and [h.k for h in hdrs[1]] == ks
        for g, o, f in zip(gs, outs, first):
            assert torch.equal(o, f)
            kept = o != 0
            assert bool((torch.sign(o[kept]) == torch.sign(g[kept].view_as(o[kept]))).all())
    a.close()


@pytest.mark.parametrize("n", [1, 3, 4097, 1_000_003])
def test_lq_budget_lengths(atomo, n):
    import torch
    g = np.random.default_rng(n).laplace(size=n).astype(np.float32)
    t = torch.from_numpy(g).cuda()
    x = np.abs(g.astype(np.float64))
    for q, want in ((2.0, x.sum() / np.sqrt((x * x).sum())), (float("inf"), x.sum() / x.max()), (3.0, x.sum() / (x ** 3).sum() ** (1 / 3))):
        got = atomo.atomo_lq_budget([t], q)
        assert abs(float(np.asarray(got).ravel()[0]) - want) <= 1e-9 * want
