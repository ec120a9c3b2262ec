"""An entry-wise encode and decode captured once in a CUDA graph and replayed, again and again and between ordinary calls: the
counters that a vector's CTAs meet at have to be as the launch itself left them, not as the host counted its launches."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("form", [0, 1, 2])                     # one kernel, two kernels, one kernel without the list
@pytest.mark.parametrize("lengths,s", [([3_000_001], 20_000.0), ([3_000_001], 400_000.0), ([70_000, 5, 900_001, 4097], 3_000.0)])
def test_replayed_capture_equals_calls(form, lengths, s):
    import torch
    from paper_1806_04090_b200 import api
    a, b = api.Atomo(0), api.Atomo(0)
    k_cap = int(s + 8 * s ** 0.5 + 8)
    size = api.payload_bytes_entrywise(lengths, k_cap)
    rng = np.random.default_rng(5)
    inputs = [[torch.from_numpy(rng.laplace(size=n).astype(np.float32)).cuda() for n in lengths] for _ in range(3)]
    wants = []
    for gs in inputs:
        b.set_entrywise_launch(form)
        buf = torch.zeros(size, dtype=torch.uint8, device="cuda")
        pay, _ = b.atomo_encode_entrywise(gs, s, seed=9, step=2, k_cap=k_cap, payload=buf)
        wants.append((buf.clone(), [o.clone() for o in b.atomo_decode(pay)]))
        assert all(h.status == 0 and h.k > 0 for h in pay.headers()[1])
    a.set_entrywise_launch(form)
    held = [g.clone() for g in inputs[0]]
    buf = torch.zeros(size, dtype=torch.uint8, device="cuda")
    outs = [torch.empty(n, device="cuda") for n in lengths]

    def step():
        pay, _ = a.atomo_encode_entrywise(held, s, seed=9, step=2, k_cap=k_cap, payload=buf)
        a.atomo_decode(pay, out=outs)

    step()                                                      # the workspace has its size before the capture
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        step()
    for turn in range(9):
        i = turn % 3
        for h, g in zip(held, inputs[i]):
            h.copy_(g)
        buf.zero_()
        step() if turn in (4, 5, 7) else graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(buf, wants[i][0]), f"turn {turn}"
        for o, w in zip(outs, wants[i][1]):
            assert torch.equal(o, w)
    del graph
    a.close()
    b.close()
