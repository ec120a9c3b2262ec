"""Layers of up to 512 rows that the TF32 Gram kernel cannot take: which of the two other kernels they go to (by the stage's launches),
and the singular values of either against 64 bits."""
import numpy as np
import pytest
import torch

from paper_1806_04090_b200 import api

pytestmark = pytest.mark.gpu

FMA, ROWS, TALL = 3, 5, 6        # launches: trace, scaling, FMA tiles | digits by rows, integer tiles, coarse tiles | digits in two passes


# short side, long side, layers.  Many narrow layers: the integer kernel's CTA per tile and its further launches cost more than they save
@pytest.mark.parametrize("r,length,count,rows,tall", [
    (16, 5001, 1, FMA, FMA), (17, 319, 1, FMA, FMA), (17, 321, 1, ROWS, FMA), (64, 447, 1, ROWS, FMA), (64, 449, 1, ROWS, TALL),
    (65, 319, 1, FMA, FMA), (65, 321, 1, ROWS, FMA), (65, 399, 1, ROWS, FMA), (65, 401, 1, ROWS, TALL), (20, 65537, 1, FMA, FMA),
    (33, 321, 32, ROWS, FMA), (33, 321, 33, FMA, FMA), (17, 511, 64, FMA, FMA), (17, 513, 64, ROWS, TALL), (17, 513, 65, FMA, FMA),
    (33, 513, 128, ROWS, TALL), (33, 513, 129, FMA, FMA), (33, 1985, 129, FMA, FMA), (33, 1987, 129, ROWS, TALL),
    (33, 257, 200, FMA, FMA), (20, 301, 200, FMA, FMA)])
def test_kernel_by_size_and_number(r, length, count, rows, tall):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(r + 5 * length)
    G = torch.randn(r, length, device="cuda", generator=gen)
    lam = torch.linalg.svdvals(G.double()).cpu().numpy() ** 2
    a = api.Atomo(0)
    a.set_profiling(True)
    for launches, layer in ((rows, G), (tall, G.T.contiguous())):
        pay, dbg = a.atomo_encode_spectral([layer] * count, 2.0, seed=3, step=0, k_cap=16, debug=True)
        assert a.stage_times()[1]["gram"] == launches
        assert all(h.status == 0 for h in pay.headers()[1])
        for l in {0, count - 1}:
            s = dbg.layer_sigma(l, r).astype(np.float64)
            # rounding A's entries to fp32 moves an eigenvalue by at most 2^-24 ||A||_F; the reduction and the sums by as much again, each
            assert np.abs(s ** 2 - lam).max() <= 4.0 * 2.0 ** -24 * np.linalg.norm(lam)
    a.close()


# short layers go along where others take the integer kernel; many narrow ones do not
@pytest.mark.parametrize("shape,count,launches", [((150, 193), 1, ROWS), ((150, 191), 1, ROWS + 1), ((33, 193), 32, ROWS), ((33, 191), 32, ROWS + 1), ((33, 193), 33, ROWS + 1),
                                                  ((90, 193), 40, ROWS), ((16, 301), 1, ROWS + 1)])
def test_short_layers_beside_others(shape, count, launches):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(sum(shape))
    short, large = (torch.randn(*s, device="cuda", generator=gen) for s in (shape, (513, 701)))
    a = api.Atomo(0)
    a.set_profiling(True)
    pay, dbg = a.atomo_encode_spectral([large] + [short] * count, 2.0, seed=3, step=0, k_cap=16, debug=True)
    assert a.stage_times()[1]["gram"] == launches
    assert all(h.status == 0 for h in pay.headers()[1])
    for l, G in ((0, large), (1, short), (count, short)):
        lam = torch.linalg.svdvals(G.double()).cpu().numpy() ** 2
        s = dbg.layer_sigma(l, min(G.shape)).astype(np.float64)
        assert np.abs(s ** 2 - lam).max() <= 4.0 * 2.0 ** -24 * np.linalg.norm(lam)
    a.close()
