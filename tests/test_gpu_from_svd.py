"""Everything downstream of the SVD, isolated: the CUDA path is given the oracle's own singular values and short-side
vectors (atomo_encode_spectral_from_svd) and must then reproduce the oracle's probabilities, masks, kept ranks,
weights and decoded gradient -- with no eigen-solver, and so no conditioning of the SVD, in between."""
import numpy as np
import pytest

from paper_1806_04090_b200 import synth
from tests import golden_io, parity

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def atomo():
    import torch
    from paper_1806_04090_b200 import api
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    a = api.Atomo(0)
    yield a
    a.close()


def _downstream(atomo, oracle, G, U, sigma, V, s, seed, step, tag):
    import torch
    m, n = G.shape
    r = min(m, n)
    short = (U if m <= n else V)                       # (short side) x r, column i = vector of atom i
    sig32 = sigma.astype(np.float32)
    enc = oracle.encode_spectral_from_svd(U, sig32.astype(np.float64), V, s, seed, step=step, layer=0)
    t = torch.from_numpy(G).cuda()
    pay, dbg = atomo.atomo_encode_spectral_from_svd([t], [torch.from_numpy(sig32).cuda()],
                                                    [torch.from_numpy(np.ascontiguousarray(short.T.astype(np.float32))).cuda()],
                                                    s, seed, step=step, k_cap=64)
    hdrs = pay.headers()
    assert hdrs[1][0].status == 0
    p = dbg.layer_prob(0, r); mask = dbg.layer_mask(0, r)
    assert np.abs(p - enc["p"]).max() <= 2e-7, f"{tag}: p {np.abs(p - enc['p']).max():.2e}"
    near = parity.near_threshold(enc)
    assert not np.any((mask != enc["mask"]) & ~near)
    arr = pay.layer_arrays(0, hdrs)
    if not np.array_equal(mask, enc["mask"]):
        return 0
    assert np.array_equal(arr["idx"], enc["idx"].astype(np.uint32))
    # weights: sigma_i / p_i with sigma_i the norm of the back-projection of the given vector
    assert parity.rel(arr["coef"], enc["coef"]) <= 1e-5
    out = atomo.atomo_decode(pay)[0].cpu().numpy().astype(np.float64)
    ref = oracle.decode_spectral(enc["coef"], enc["U_S"], enc["V_S"])
    if enc["idx"].size:
        assert parity.rel(out, ref) <= parity.REL_TOL, f"{tag}: decode {parity.rel(out, ref):.2e}"
    else:
        assert not out.any()
    return 1


@pytest.mark.parametrize("shape", [(64, 64), (64, 576), (300, 130), (512, 2304)])
def test_downstream_of_the_oracle_svd(atomo, oracle, shape):
    G = synth.lowrank_plus_noise(np.random.default_rng([3, *shape]), shape[0], shape[1], 1.0, noise_rel=0.01)
    U, sigma, V = oracle.jacobi_svd(G)
    done = 0
    for s, seed in ((2.0, 5), (3.5, 6), (8.0, 7)):
        done += _downstream(atomo, oracle, G, U, sigma, V, s, seed, 1, f"{shape} s={s}")
    assert done > 0                                     # at least one budget was compared to the end


def test_downstream_of_a_library_svd_at_1024(atomo, oracle):
    # short side 1024 (config-5 shape): the oracle's SVD takes minutes there; a library SVD in fp64 gives the same
    # decomposition to 1e-12 (checked for the stored cases in the CPU tests) and is what is handed to both sides
    G = synth.c5_stress_layer(0, 0)
    U, sigma, Vt = np.linalg.svd(G.astype(np.float64), full_matrices=False)
    assert _downstream(atomo, oracle, G, U, sigma, Vt.T, 4.0, 11, 2, "1024 x 4096") == 1


def test_atom_of_subnormal_norm(atomo):
    """A given vector that meets the layer's rows in a subnormal entry only: its atom contributes nothing, and nothing that is not finite."""
    import torch
    G = torch.zeros(8, 64, device="cuda")
    G[0] = torch.linspace(-2.0, 2.0, 64, device="cuda")
    short = torch.eye(8, device="cuda")
    short[1:, 0] = 1.0e-41
    pay, _ = atomo.atomo_encode_spectral_from_svd([G], [torch.full((8,), 1.0, device="cuda")], [short], 8.0, 3, step=1, k_cap=8)
    assert pay.headers()[1][0].status == 0 and pay.headers()[1][0].k == 8
    assert np.isfinite(pay.layer_arrays(0)["V"]).all()
    out = atomo.atomo_decode(pay)[0]
    assert float((out - G).abs().max()) <= 2.0 ** -22 * 2.0
