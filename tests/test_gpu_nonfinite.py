"""Alpha-profile plans on signals with a NaN or infinite sample: every bin of such a signal's estimate is NaN,
and the profile says so under every schedule (a zero profile would read as silence); the other signals
of the plan are untouched, and the next run on clean samples is clean again."""
import pytest

from paper_2506_18003_gb300 import binding, signals

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    import torch as t
    assert t.cuda.is_available(), "GPU tests need CUDA"
    binding.load()
    return t


def _profile(torch, plan, x, power):
    plan.set_output("profile", power)
    out = torch.full((plan.out_offsets[-1],), -1.0, dtype=torch.float32, device="cuda")
    plan.run(x, out, torch.empty(max(1, plan.workspace_bytes), dtype=torch.uint8, device="cuda"))
    binding.scd_check_device()
    return [plan.output(out, i).clone() for i in range(plan.nsig)]


@pytest.mark.parametrize("estimator,Np,L", [("ssca", 16, 1), ("ssca", 64, 1), ("ssca", 256, 1), ("fam", 32, 8)])
@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
@pytest.mark.parametrize("power", [1, 2])
def test_profile_of_nonfinite_signal(torch, estimator, Np, L, bad, power):
    lengths = [4096, 8192, 8192]
    x = torch.cat([torch.from_numpy(signals.batch_signal(700 + i, n)) for i, n in enumerate(lengths)]).cuda()
    dirty = x.clone()
    dirty[4096 + 1234] = complex(bad, 1.0)
    got = {}
    for sched in ("auto", "stages", "persistent"):
        plan = binding.BatchPlan(estimator, lengths, Np, L)
        plan.set_schedule(sched)
        clean = _profile(torch, plan, x, power)
        got[sched] = _profile(torch, plan, dirty, power)
        for i in (0, 2):
            assert torch.equal(got[sched][i], clean[i]), (sched, i)
        for a, b in zip(_profile(torch, plan, x, power), clean):
            assert torch.equal(a, b), sched
        plan.close()
    want = ~torch.isfinite(got["persistent"][1])
    assert bool(want.any())
    for sched in ("auto", "stages"):
        assert torch.equal(~torch.isfinite(got[sched][1]), want), sched
        if bad != bad:                                       # NaN in, NaN out
            assert torch.equal(torch.isnan(got[sched][1]), torch.isnan(got["persistent"][1])), sched
