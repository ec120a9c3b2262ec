"""The calls whose speed counts, as a data-parallel training step makes them: every worker encodes its layer gradients
(spectral or entry-wise atoms) into a payload and decodes payloads back to dense gradients.

`listed()` gives fixed cases, `draw(rng)` more of the same ranges, `prepare` what a training program holds before the call
(gradients, payload and output buffers, the library context) and `run` one pass through the public entry points.

Inputs: a layer's gradient is a few directions with singular values i^-decay under the sampling noise of a worker's share
of the mini-batch, whose Frobenius norm is `noise` times that of the signal: a few dominant singular values above a broad
bulk.  Entry-wise gradients are Laplace(0, 1e-3), or N(0, 1) for the small vector.
"""
import math

import torch

from paper_1806_04090_b200 import api, synth

SIGNAL_RANK = 16


def _set(layers):
    return ",".join("%dx%d" % (l.rows, l.cols) for l in layers)


def _lengths(layers):
    return ",".join("%d" % (l.rows * l.cols) for l in layers)


def listed():
    return [
        # one small layer: nothing but launches, dependent steps and the host's part of the call
        {"name": "spectral_64x64", "kind": "spectral", "shapes": "64x64", "s": 2.0, "decay": 1.0, "noise": 4.0},
        # every layer of a CIFAR ResNet-18 in one call: the ordinary training step (Table 2 of the paper)
        {"name": "spectral_resnet18", "kind": "spectral", "shapes": _set(synth.RESNET18_LAYERS), "s": 2.0, "decay": 1.5, "noise": 4.0},
        # VGG-11 with two 4096 x 4096 fully connected layers: one or two layers outweigh all others
        {"name": "spectral_vgg11", "kind": "spectral", "shapes": _set(synth.VGG11_LAYERS), "s": 3.0, "decay": 1.0, "noise": 4.0},
        # many equal layers of a wide model: throughput with the GPU full
        {"name": "spectral_96x1024x4096", "kind": "spectral", "shapes": "96*1024x4096", "s": 4.0, "decay": 1.0, "noise": 4.0},
        # what no tile divides: odd short sides, layers taller than wide, the paper's own tall reshape of a convolution
        {"name": "spectral_ragged", "kind": "spectral", "shapes": "777x3001,1023x515,333x1000,129x4097,2047x255,65x65,16384x18,96x18,30x4000",
         "s": 3.0, "decay": 1.0, "noise": 4.0},
        # one small vector: launches and the host's part of the call
        {"name": "entrywise_4096", "kind": "entrywise", "lengths": "4096", "s": 64.0, "values": "normal", "format": "explicit", "qsgd": False},
        # every layer of the ResNet-18 as a vector of its own, the same budget for each (the smallest are kept whole)
        {"name": "entrywise_resnet18_layers", "kind": "entrywise", "lengths": _lengths(synth.RESNET18_LAYERS), "s": 6100.0,
         "values": "laplace", "format": "explicit", "qsgd": False},
        # a whole model's gradient as one vector at the ordinary budget of 1 %
        {"name": "entrywise_25m_1pct", "kind": "entrywise", "lengths": "25600000", "s": 256000.0, "values": "laplace", "format": "explicit", "qsgd": False},
        # unbiased l2 quantisation (Section 4): budget ||g||_1 / ||g||_2, compact payload, every step with its own budget
        {"name": "entrywise_25m_qsgd", "kind": "entrywise", "lengths": "25600000", "s": 0.0, "values": "laplace", "format": "compact", "qsgd": True},
        # a large model at a large budget, of odd length
        {"name": "entrywise_100m_10pct", "kind": "entrywise", "lengths": "100000001", "s": 10000000.0, "values": "laplace", "format": "explicit", "qsgd": False},
        # the receiving side of a step: the mean of eight workers' payloads
        {"name": "average_8_resnet18", "kind": "average_spectral", "shapes": _set(synth.RESNET18_LAYERS), "s": 3.0, "decay": 1.5, "noise": 4.0, "workers": 8},
        {"name": "average_8_entrywise_25m", "kind": "average_entrywise", "lengths": "25600000", "s": 256000.0, "values": "laplace",
         "format": "explicit", "workers": 8},
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["spectral", "spectral", "stack", "entrywise", "entrywise", "entrywise_layers", "average_spectral", "average_entrywise"])
    if kind in ("spectral", "stack", "average_spectral"):
        base = {"s": round(rng.uniform(1.0, 8.0), 2), "decay": round(rng.uniform(1.0, 1.5), 2), "noise": round(rng.uniform(3.0, 8.0), 2)}
        if kind == "stack":   # equal layers, at most 2e8 elements in all
            r = int(_log(rng, 32, 1500))
            length = int(_log(rng, r, 8192))
            count = max(2, min(int(_log(rng, 2, 120)), int(2.0e8 / (r * length))))
            return dict(base, kind="spectral", shapes="%d*%dx%d" % (count, r, length))
        shapes, total, cubes = [], 0, 0.0
        for _ in range(rng.randint(1, 16)):
            r = int(_log(rng, 10, 2400))
            length = int(_log(rng, r, 8192))
            if total + r * length > 1.0e8 or cubes + float(r) ** 3 > 6.0e10:
                r, length = int(_log(rng, 10, 300)), int(_log(rng, 300, 3000))
            total, cubes = total + r * length, cubes + float(r) ** 3
            shapes.append("%dx%d" % ((length, r) if rng.random() < 0.25 else (r, length)))
        case = dict(base, kind=kind, shapes=",".join(shapes))
        if kind == "average_spectral":
            case["workers"] = rng.randint(2, 16)
        return case
    frac = _log(rng, 1e-3, 0.1)
    case = {"kind": kind.replace("_layers", ""), "values": "laplace", "format": rng.choice(["explicit", "explicit", "compact"])}
    if kind == "entrywise_layers":
        lengths = [int(_log(rng, 1e3, 5e6)) for _ in range(rng.randint(2, 20))]
    else:
        lengths = [int(_log(rng, 1e3, 1e8 if kind == "entrywise" else 3e7))]
    case["lengths"] = ",".join("%d" % n for n in lengths)
    case["s"] = round(max(2.0, frac * sum(lengths) / len(lengths)), 1)
    if kind == "average_entrywise":
        case["workers"] = rng.randint(2, 16)
    else:
        case["qsgd"] = len(lengths) == 1 and case["format"] == "compact" and rng.random() < 0.5
        if case["qsgd"]:
            case["s"] = 0.0
    return case


# ---- sizes --------------------------------------------------------------------------------------
def _shapes(case):
    out = []
    for part in case["shapes"].split(","):
        count, _, shape = part.rpartition("*")
        rows, cols = shape.split("x")
        out += [(int(rows), int(cols))] * int(count or 1)
    return out


def _vec_lengths(case):
    return [int(x) for x in case["lengths"].split(",")]


def _qsgd_budget(n):
    return math.sqrt(0.5 * n)      # ||g||_1 / ||g||_2 of n Laplace entries


def _budget(case):
    return _qsgd_budget(_vec_lengths(case)[0]) if case.get("qsgd") else case["s"]


# ---- inputs -------------------------------------------------------------------------------------
def _layer(m, n, case, gen, dev):
    q = min(m, n, SIGNAL_RANK)
    sigma = torch.arange(1, q + 1, dtype=torch.float32, device=dev) ** (-case["decay"])
    u = torch.randn(m, q, device=dev, generator=gen) / math.sqrt(m)
    v = torch.randn(n, q, device=dev, generator=gen) / math.sqrt(n)
    g = torch.randn(m, n, device=dev, generator=gen)
    g *= case["noise"] * float(torch.linalg.norm(sigma)) / math.sqrt(m * n)
    return g.addmm_(u * sigma, v.T)


def _vector(n, case, gen, dev):
    if case["values"] == "normal":
        return torch.randn(n, device=dev, generator=gen)
    u = torch.rand(n, device=dev, generator=gen).sub_(0.5)
    return torch.log1p(u.abs().mul_(-2.0).clamp_(min=-0.9999999)).mul_(-1.0e-3).copysign_(u)


_contexts = {}


def _context(compact=False):
    """One library context per payload format for the whole program, as a training loop keeps it."""
    if compact not in _contexts:
        a = api.Atomo(0)
        if compact:
            a.set_entrywise_format(api.EW_COMPACT, sat_cap=1 << 16)
        _contexts[compact] = a
    return _contexts[compact]


def _align(x):
    return (x + 15) // 16 * 16


def _wire_views(pay, kind, shapes, k_cap, compact):
    """Views of what a payload buffer says besides the vectors: per layer (k_cap, k, saturated, status), and the arrays of
    kept indices and their values (spectral: ranks and coefficients)."""
    n = len(shapes)
    words = pay.view(torch.int32)
    views = {"counts": words.as_strided((n, 4), (20, 1), 20)}
    offsets, off = [], 64 + 80 * n
    for rows, cols in shapes:
        first = off = _align(off)
        if kind == api.KIND_SPECTRAL:
            r, length = min(rows, cols), max(rows, cols)
            kc = min(k_cap, r)
            second = _align(off + 4 * kc)
            off = _align(_align(second + 4 * kc) + 4 * kc * r) + 4 * kc * length
        else:
            kc, sat = min(k_cap, cols), min(1 << 16, cols) if compact else 0
            second = _align(off + (2 if compact else 4) * kc)
            off = _align(second + 4 * (sat if compact else kc)) + 4 * ((cols + api.EW_TILE - 1) // api.EW_TILE + 1)
            off = _align(off) + 4 * sat
        offsets.append((first, second, kc, kc if not compact else sat))
    f32 = pay.view(torch.float32)
    if n > 24:                          # equal layers: one strided view for all of them
        step = (offsets[1][0] - offsets[0][0]) // 4
        first, second, kc, _ = offsets[0]
        views["idx"] = words.as_strided((n, kc), (step, 1), first // 4)
        views["val"] = f32.as_strided((n, kc), (step, 1), second // 4)
        return views
    ent = pay.view(torch.int16) if compact else words
    size = 2 if compact else 4
    views["idx"] = [ent[a // size: a // size + c] for a, _, c, _ in offsets]
    views["val"] = [f32[b // 4: b // 4 + c] for _, b, _, c in offsets]
    return views


def prepare(case, seed):
    dev = torch.device("cuda", 0)
    gen = torch.Generator(device=dev)
    gen.manual_seed(int(seed))
    spectral = case["kind"].endswith("spectral")
    compact = case.get("format") == "compact"
    a = _context(compact)
    workers = case.get("workers", 0)
    if spectral:
        shapes = _shapes(case)
        k_cap = api.default_k_cap(case["s"], max(min(x) for x in shapes))
        size = api.payload_bytes_spectral(shapes, k_cap)
    else:
        lengths = _vec_lengths(case)
        shapes = [(1, n) for n in lengths]
        k_cap = api.default_k_cap(1.05 * _budget(case) if case.get("qsgd") else case["s"], max(lengths))
        size = api.payload_bytes_entrywise_compact(lengths, k_cap, 1 << 16) if compact else api.payload_bytes_entrywise(lengths, k_cap)

    def gradients():
        if spectral:
            return [_layer(m, n, case, gen, dev) for m, n in shapes]
        return [_vector(n, case, gen, dev) for n in lengths]

    flat = torch.zeros(sum(m * n for m, n in shapes), dtype=torch.float32, device=dev)
    outs, at = [], 0
    for m, n in shapes:
        outs.append(flat[at: at + m * n].view((m, n) if spectral else (n,)))
        at += m * n
    state = {"a": a, "s": case["s"], "seed": int(seed) % (1 << 31), "step": int(seed) % 1000, "k_cap": k_cap, "flat": flat, "outs": outs,
             "spectral": spectral, "workers": workers, "qsgd": bool(case.get("qsgd"))}
    if not workers:
        buf = torch.zeros(size, dtype=torch.uint8, device=dev)
        state.update(grads=gradients(), buf=buf, wire=_wire_views(buf, api.KIND_SPECTRAL if spectral else api.KIND_ENTRYWISE, shapes, k_cap, compact))
        return state
    # the payloads of all workers, as an all-gather leaves them
    encode = a.atomo_encode_spectral if spectral else a.atomo_encode_entrywise
    pays = []
    for w in range(workers):
        buf = torch.zeros(size, dtype=torch.uint8, device=dev)
        pays.append(encode(gradients(), case["s"], state["seed"] + w, step=state["step"], k_cap=k_cap, payload=buf)[0])
    state["payloads"] = pays
    return state


def run(state):
    a = state["a"]
    if state["workers"]:
        a.atomo_decode_average(state["payloads"], out=state["outs"])
        return {"mean": state["flat"]}
    s = state["s"]
    if state["spectral"]:
        pay, _ = a.atomo_encode_spectral(state["grads"], s, state["seed"], step=state["step"], k_cap=state["k_cap"], payload=state["buf"])
    else:
        if state["qsgd"]:
            s = a.atomo_lq_budget(state["grads"], 2.0)[0]
        pay, _ = a.atomo_encode_entrywise(state["grads"], s, state["seed"], step=state["step"], k_cap=state["k_cap"], payload=state["buf"])
    a.atomo_decode(pay, out=state["outs"])
    return {"decoded": state["flat"], "wire": state["wire"]}


# ---- what a pass cannot do without ----------------------------------------------------------------
def work(case):
    workers = case.get("workers", 0)
    if case["kind"].endswith("spectral"):
        moved = flops = 0.0
        for m, n in _shapes(case):
            r, k = min(m, n), min(case["s"], min(m, n))
            payload = 4.0 * k * (m + n + 2)
            if workers:
                moved += 4.0 * m * n + workers * payload
                flops += 2.0 * workers * k * m * n
            else:   # gradient in, payload out; payload in, gradient out
                moved += 8.0 * m * n + 2.0 * payload
                # Gram product on the short side, reduction to tridiagonal form, back-projection and decode of k atoms
                flops += float(r) * m * n + 4.0 / 3.0 * float(r) ** 3 + 4.0 * k * m * n
        return {"bytes": moved, "flops": flops}
    moved = flops = 0.0
    for n in _vec_lengths(case):
        k = min(_budget(case), n)
        payload = (2.0 if case["format"] == "compact" else 8.0) * k
        if workers:
            moved += 4.0 * n + workers * payload
            flops += workers * k
        else:
            moved += 8.0 * n + 2.0 * payload
            flops += 4.0 * n + (2.0 * n if case.get("qsgd") else 0.0)
    return {"bytes": moved, "flops": flops}


def tolerance(case):
    if not case["kind"].endswith("spectral"):
        # sums in 64 bits, values in 32: indices and counts are the same
        return {"rel": 1e-5, "differ": 0.0}
    # A kept atom's vectors move by the rounding of the fp32 Gram matrix and of its reduction over the distance to the
    # next squared singular value; in the noise bulk that distance is 1e-4 ... 1e-6 of the largest one, on average, and
    # shrinks with the short side.  (Other summation orders of the same precision gave up to 6e-5.)
    wide = max(min(x) for x in _shapes(case)) > 512
    return {"rel": 2e-3 if wide else 2e-4, "max": 0.1 if wide else 0.02, "differ": 0.0}
