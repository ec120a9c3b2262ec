"""Small and large layers in one call run partly side by side: what each yields must not depend on that, on the stream, or on a replay
from a graph.  (The sets are chosen such that every layer takes the same kernels with and without the others; the last digits may
depend on the company where that is not so.)"""
import pytest
import torch

from paper_1806_04090_b200 import api

pytestmark = pytest.mark.gpu


def _layers():
    gen = torch.Generator(device="cuda")
    gen.manual_seed(4)
    return [torch.randn(m, n, device="cuda", generator=gen) for m, n in ((40, 90), (300, 500), (512, 700), (1100, 1300), (600, 650))]


def _arrays(pay, n):
    return [{k: v.copy() for k, v in pay.layer_arrays(l).items() if hasattr(v, "copy")} for l in range(n)]


def test_small_layers_beside_large_ones():
    G = _layers()
    a = api.Atomo(0)
    # (draws are by a layer's place in its call: for their vectors the large ones stand behind layers next to which nothing runs for long)
    alone, _ = a.atomo_encode_spectral(G[:3], 3.0, seed=9, step=2, k_cap=24)
    want = _arrays(alone, 3)
    tiny = [torch.ones(1, 1, device="cuda")] * 3
    large, _ = a.atomo_encode_spectral(tiny + G[3:], 3.0, seed=9, step=2, k_cap=24)
    want += _arrays(large, 5)[3:]
    _, dbg = a.atomo_encode_spectral(G[3:], 3.0, seed=9, step=2, k_cap=24, debug=True)
    sigma = [dbg.layer_sigma(l, min(G[3 + l].shape)).copy() for l in range(2)]
    for stream in (torch.cuda.current_stream(), torch.cuda.Stream(), torch.cuda.Stream()):
        stream.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(stream):
            pay, _ = a.atomo_encode_spectral(G, 3.0, seed=9, step=2, k_cap=24)
            out = a.atomo_decode(pay)
        stream.synchronize()
        assert [h.status for h in pay.headers()[1]] == [0] * 5
        for x, y in zip(want, _arrays(pay, 5)):
            assert x.keys() == y.keys()
            assert all((x[k] == y[k]).all() for k in x)
        assert all(torch.isfinite(o).all() for o in out)
    _, dbg = a.atomo_encode_spectral(G, 3.0, seed=9, step=2, k_cap=24, debug=True)
    assert all((dbg.layer_sigma(3 + l, min(G[3 + l].shape)) == sigma[l]).all() for l in range(2))
    a.close()


def test_replay_from_a_graph():
    G = _layers()
    a = api.Atomo(0)
    shapes = [tuple(g.shape) for g in G]
    buf = torch.zeros(api.payload_bytes_spectral(shapes, 24), dtype=torch.uint8, device="cuda")
    stream = torch.cuda.Stream()
    stream.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(stream):                    # (the tables are uploaded on the stream that is captured later)
        a.atomo_encode_spectral(G, 3.0, seed=9, step=2, k_cap=24, payload=buf)
    torch.cuda.synchronize()
    want = buf.clone()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        a.atomo_encode_spectral(G, 3.0, seed=9, step=2, k_cap=24, payload=buf)
    for _ in range(3):
        buf.zero_()
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(buf, want)
    del graph
    a.close()


@pytest.mark.parametrize("priority", [0, -1])
def test_side_stream_has_the_callers_priority(priority):
    from cuda.bindings import runtime as rt
    G = _layers()
    a = api.Atomo(0)
    buf = torch.zeros(api.payload_bytes_spectral([tuple(g.shape) for g in G], 24), dtype=torch.uint8, device="cuda")
    stream = torch.cuda.Stream(priority=priority)
    other = torch.cuda.Stream(priority=-1 - priority)
    for st in (stream, other):                         # the context has seen calls of either kind (tables: see above)
        st.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(st):
            a.atomo_encode_spectral(G, 3.0, seed=9, step=2, k_cap=24, payload=buf)
        torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(graph, stream=stream):
        a.atomo_encode_spectral(G, 3.0, seed=9, step=2, k_cap=24, payload=buf)
    raw = rt.cudaGraph_t(init_value=graph.raw_cuda_graph())
    err, _, n = rt.cudaGraphGetNodes(raw, 0)
    err, nodes, n = rt.cudaGraphGetNodes(raw, n)
    seen = []
    for node in nodes[:n]:
        err, kind = rt.cudaGraphNodeGetType(node)
        if kind == rt.cudaGraphNodeType.cudaGraphNodeTypeKernel:
            err, value = rt.cudaGraphKernelNodeGetAttribute(node, rt.cudaLaunchAttributeID.cudaLaunchAttributePriority)
            assert err == rt.cudaError_t.cudaSuccess
            seen.append(value.priority)
    assert len(seen) >= 10 and set(seen) == {stream.priority}
    del graph
    a.close()
