"""Stage timers of the entry-wise encode: the solve of the two-kernel form has a stage of its own."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("form,solves,packs", [(0, 0, 1), (1, 2, 2), (2, 0, 1)])
def test_solve_and_pack_are_timed_apart(form, solves, packs):
    import torch
    from paper_1806_04090_b200 import api
    a = api.Atomo(0)
    a.set_entrywise_launch(form)
    gs = [torch.randn(n, device="cuda") for n in (500_000, 70_001)]
    a.set_profiling(True)
    a.atomo_encode_entrywise(gs, 2000.0, seed=1, step=1)
    ms, launches = a.stage_times()
    assert (launches["ew_reduce"], launches["ew_pack"]) == (solves, packs)
    assert (ms["ew_reduce"] > 0) == (solves > 0) and ms["ew_pack"] > 0
    a.close()
