"""The instances of the entry-wise encode (chunks in registers, with a candidate list, with a list of large atoms, mixed) around the
sizes where one gives way to the next, against the two-kernel form."""
import numpy as np
import pytest
import torch

from paper_1806_04090_b200 import api

pytestmark = pytest.mark.gpu

TILE, SMS = 4096, 148


@pytest.fixture(scope="module")
def atomo():
    a = api.Atomo(0)
    yield a
    a.close()


# one tile per chunk, chunks of four tiles (registers), of four and five (mixed), of five and more
@pytest.mark.parametrize("n", [1, TILE - 1, 3 * TILE + 1, 4 * SMS * TILE, 4 * SMS * TILE + 1, 5 * SMS * TILE, 9 * SMS * TILE - 5])
@pytest.mark.parametrize("frac", [0.003, 0.2])
def test_kinds_against_two_kernels(atomo, n, frac):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(n % 1000003)
    g = torch.randn(n, device="cuda", generator=gen) ** 3      # some atoms with p = 1 at the larger budget
    s = max(1.0, frac * n)
    got = []
    try:
        for form, debug in ((0, "mask"), (0, True), (2, True), (1, True)):   # (probabilities asked for: no list, no registers)
            atomo.set_entrywise_launch(form)
            pay, dbg = atomo.atomo_encode_entrywise([g], s, seed=11, step=4, k_cap=int(1.2 * s) + 2000, debug=debug)
            head = pay.headers()[1][0]
            assert head.status == 0
            got.append((head.k, head.n_sat, dbg.mask_words.clone(), pay.layer_arrays(0)["idx"].copy(), atomo.atomo_decode(pay)[0].clone()))
    finally:
        atomo.set_entrywise_launch(0)
    for other in got[1:]:
        assert other[:2] == got[0][:2] and torch.equal(other[2], got[0][2]) and np.array_equal(other[3], got[0][3])
        # (sum |g| depends on the cut at the 1e-8 level, the weights are its fp32 roundings)
        assert float((other[4] - got[0][4]).norm()) <= 1e-6 * float(got[0][4].norm())


def test_several_short_vectors_and_a_long_one(atomo):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(3)
    short = [torch.randn(n, device="cuda", generator=gen) for n in (5, 4096, 16384, 16385)]
    long = torch.randn(6 * SMS * TILE, device="cuda", generator=gen)
    for vecs in (short, short + [long]):                       # all in registers, mixed
        pay, dbg = atomo.atomo_encode_entrywise(vecs, 50.0, seed=11, step=4, k_cap=400, debug=True)
        outs = atomo.atomo_decode(pay)
        for l, v in enumerate(vecs[:4]):
            head = pay.headers()[1][l]
            assert head.status == 0 and head.k == np.count_nonzero(dbg.layer_mask(l, v.numel()))
            kept = outs[l] != 0
            p = torch.from_numpy(dbg.layer_prob(l, v.numel())).cuda()
            assert torch.allclose(outs[l][kept], v[kept] / p[kept], rtol=1e-5)
