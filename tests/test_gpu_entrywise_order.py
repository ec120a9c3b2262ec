"""The sums of the water-filling rounds have a fixed order: a call gives the same payload every time.

The vector is made so that the order shows.  Each of its 256 runs (the 16 entries a lane takes of a unit) holds one entry H = 2^23 that
saturates in the first round; the sum T of what is left then decides the weight c = T / 4.  One run leaves 2^24, one nearly 1 and
the others multiples of 2^-30, a few of fp64's last places at 2^24, and together they are 2^24 + 1, half way between two fp32 numbers:
any order of additions gives T within ten roundings of that (the sum of a tree of ten levels), and c lands above or below with it."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _vector(seed):
    rng = np.random.default_rng(seed)
    tiny = rng.integers(1, 8, size=254) * 2.0 ** -30
    near_one = 1.0 - float(np.ceil(tiny.sum() * 2.0 ** 24) * 2.0 ** -24)     # an fp32 number below 1
    tiny[0] += 1.0 - near_one - tiny.sum()                                   # the exact total of both is 1
    runs = np.zeros((256, 16), dtype=np.float64)
    runs[:, 5] = 2.0 ** 23
    order = rng.permutation(256)
    runs[order[0], 8:16] = 2.0 ** 21
    runs[order[1], 8] = near_one
    runs[order[2:], 9] = tiny
    assert runs.sum() - 256 * 2.0 ** 23 == 2.0 ** 24 + 1 and np.array_equal(runs, runs.astype(np.float32))
    return runs.reshape(256, 4, 4).transpose(1, 0, 2).reshape(4096).astype(np.float32)


@pytest.mark.parametrize("seed", [0, 1, 2, 3])
def test_same_payload_every_time(seed):
    import torch
    from paper_1806_04090_b200 import api
    a = api.Atomo(0)
    a.set_entrywise_launch(1)                                   # (the solve kernel lists the runs of any vector)
    g = torch.from_numpy(_vector(seed)).cuda()
    buf = torch.zeros(api.payload_bytes_entrywise([4096], 4096), dtype=torch.uint8, device="cuda")
    first = None
    for turn in range(300):
        buf.zero_()
        pay, _ = a.atomo_encode_entrywise([g], 260.0, seed=3, step=1, k_cap=4096, payload=buf)
        if first is None:
            first = buf.clone()
            h = pay.headers()[1][0]
            assert h.status == 0 and h.n_sat == 256 and abs(h.c - (2.0 ** 24 + 1) / 4) <= 0.25
        assert torch.equal(buf, first), f"turn {turn}"
    a.close()
