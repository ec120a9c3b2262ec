"""Layers of rank one: the reduction's columns shrink by the rounding unit from step to step, down to the smallest numbers."""
import pytest
import torch

from paper_1806_04090_b200 import api

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,n", [(17, 233), (30, 236), (57, 730), (70, 1373), (90, 1040), (406, 620), (1334, 99), (1931, 103), (5000, 64), (512, 513), (600, 777), (1100, 1200)])
def test_equal_entries(m, n):
    a = api.Atomo(0)
    for value in (0.37, 1.0, -3.0e-3, 0.1):
        for pad in (0, 1):                                     # either kernel of the Gram matrix
            G = torch.full((m, n + pad), value, device="cuda")[:, :n]
            pay, _ = a.atomo_encode_spectral([G], 1.0, 5, step=1, k_cap=16)
            head = pay.headers()[1][0]
            assert head.status == 0
            out = a.atomo_decode(pay)[0]
            assert torch.isfinite(out).all()
            if head.k and pay.layer_arrays(0)["idx"][0] == 0:  # (the other singular values come out at rounding level, and share the budget)
                assert float((out - G).norm()) <= 0.2 * float(G.norm())
    a.close()
