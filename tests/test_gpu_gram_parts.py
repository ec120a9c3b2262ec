"""Layers with a very long side: the K range of their Gram matrix is cut into a bounded number of parts, so that the workspace of
the partial sums does not grow with the gradient, and the sums stay right."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,n", [(1, 20_000_003), (20_000_003, 1), (3, 5_000_001), (6_000_001, 5)])
def test_workspace_and_sigma_of_long_layers(m, n):
    import torch
    from paper_1806_04090_b200 import api
    a, r = api.Atomo(0), min(m, n)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(m + n)
    G = torch.randn(m, n, device="cuda", generator=gen) * 1e-3
    buf = torch.zeros(api.payload_bytes_spectral([(m, n)], r), dtype=torch.uint8, device="cuda")
    small = torch.randn(4, 8, device="cuda")
    a.atomo_encode_spectral([small], 1.0, seed=1, k_cap=2)      # whatever the first call loads
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    pay, dbg = a.atomo_encode_spectral([G], 1.0, seed=1, step=1, k_cap=r, payload=buf, debug=True)
    torch.cuda.synchronize()
    used = free - torch.cuda.mem_get_info()[0]
    assert pay.headers()[1][0].status == 0
    X = (G if m <= n else G.T).double()
    want = torch.linalg.eigvalsh(X @ X.T).clamp(min=0).sqrt().flip(0).cpu().numpy()
    # fp32 runs of 32 products added in fp64, one rounding to fp32: a few 2^-24
    assert np.abs(dbg.layer_sigma(0, r) - want).max() <= 4 * 2.0 ** -24 * want[0]
    # the long-side vectors of up to r atoms are as large as the gradient, and the workspace is allocated with some to spare
    assert used <= 2 * 4 * m * n + (64 << 20), f"{used / (4 * m * n):.2f} times the gradient"
    a.close()
