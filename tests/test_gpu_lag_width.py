"""The channel pass of the lag domain takes wider tiles at Np = 256 where a launch writes much; a signal's estimate
must not depend on how many signals share its launch: a plan above the limit against the single calls
below it, estimates and profiles, bit for bit, and one estimate against the FP64 oracle."""
import numpy as np
import pytest

from oracle import scd_oracle as orc
from paper_2506_18003_gb300 import binding, signals

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    import torch as t
    assert t.cuda.is_available(), "GPU tests need CUDA"
    binding.load()
    return t


@pytest.mark.parametrize("N,count", [(1 << 14, 33), (1 << 16, 9)])
def test_estimates_do_not_depend_on_the_class(torch, N, count):
    Np = 256
    sigs = [signals.batch_signal(1500 + i, N) for i in range(count)]
    x = torch.from_numpy(np.concatenate(sigs)).cuda()
    plan = binding.BatchPlan("ssca", [N] * count, Np)
    ws = torch.empty(plan.workspace_bytes, dtype=torch.uint8, device="cuda")
    out = torch.empty(plan.out_offsets[-1], dtype=torch.complex64, device="cuda")
    assert out.numel() * 8 > 1 << 30
    plan.run(x, out, ws)
    binding.scd_check_device()
    for i in range(count):
        assert torch.equal(plan.output(out, i), binding.scd_ssca(x[i * N:(i + 1) * N].clone(), Np)), i
    ch = np.array([0, 1, 127, 128, 255])
    est = plan.output(out, count - 1)
    ref = orc.ssca(sigs[-1], orc.hamming_window(Np), Np, channels=ch, chunk=1 << 15)
    got = est[torch.from_numpy(ch).cuda()].cpu().numpy()
    assert float(np.max(np.abs(got - ref))) / est.abs().max().item() <= 1e-5
    same = [binding.scd_ssca_alpha_profile(plan.output(out, i), N, Np, power=1) for i in range(count)]
    plan.set_output("profile", 1)
    prof = torch.empty(plan.out_offsets[-1], dtype=torch.float32, device="cuda")
    plan.run(x, prof, ws)
    binding.scd_check_device()
    for i in range(count):
        assert torch.equal(plan.output(prof, i), same[i]), i
    plan.close()
    del out, ws
    torch.cuda.empty_cache()
