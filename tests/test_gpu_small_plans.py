"""SSCA plans whose launches weigh more than their work: one size class (direct dependent launches), several (a
graph branch per class), and both sides of the limits (one set of strip launches or two for profiles, in
a row above 128 MB).  Runs queued back to back on inputs and outputs in turn, outputs dirty: every
estimate equal to scd_ssca's and every profile to its estimate's, bit for bit."""
import pytest

from paper_2506_18003_gb300 import binding

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    import torch as t
    assert t.cuda.is_available(), "GPU tests need CUDA"
    binding.load()
    return t


@pytest.mark.parametrize("Np,lengths", [
    (64, [8192]), (64, [8192] * 3), (16, [5000] * 9), (128, [1 << 15] * 2), (64, [4096, 9000]),
    (16, [40000, 4096, 9000, 17000, 5000]), (256, [4096, 20000]), (32, [4096] * 40 + [1 << 16]),
    (64, [1 << 18, 4096]), (32, [1 << 17, 1 << 19])])
def test_small_plans(torch, Np, lengths):
    plan = binding.BatchPlan("ssca", lengths, Np)
    xs = [torch.randn(sum(lengths), dtype=torch.complex64, device="cuda") for _ in range(2)]
    ws = torch.empty(plan.workspace_bytes, dtype=torch.uint8, device="cuda")
    st = torch.cuda.Stream()
    outs = [torch.full((plan.out_offsets[-1],), 7.0, dtype=torch.complex64, device="cuda") for _ in range(2)]
    st.wait_stream(torch.cuda.current_stream())
    for i in range(6):
        plan.run(xs[i % 2], outs[i % 2], ws, stream=st)
    binding.scd_check_device(st)
    est = [[plan.output(outs[j], i).clone() for i in range(plan.nsig)] for j in range(2)]
    for j in range(2):
        for i in range(plan.nsig):
            x = xs[j][plan.x_offsets[i]:plan.x_offsets[i] + plan.sizes[i]].clone()
            assert torch.equal(est[j][i], binding.scd_ssca(x, Np)), (j, i)
    plan.set_output("profile", 1)
    outs = [torch.full((plan.out_offsets[-1],), 1e9, dtype=torch.float32, device="cuda") for _ in range(2)]
    st.wait_stream(torch.cuda.current_stream())
    for i in range(6):
        plan.run(xs[i % 2], outs[i % 2], ws, stream=st)
    binding.scd_check_device(st)
    for j in range(2):
        for i in range(plan.nsig):
            same = binding.scd_ssca_alpha_profile(est[j][i], plan.sizes[i], Np, power=1)
            assert torch.equal(plan.output(outs[j], i), same), (j, i)
    plan.close()


def test_null_stream(torch):
    """The legacy stream: direct launches of any plan."""
    lengths, Np = [4096, 9000], 32
    plan = binding.BatchPlan("ssca", lengths, Np)
    x = torch.randn(sum(lengths), dtype=torch.complex64, device="cuda")
    ws = torch.empty(plan.workspace_bytes, dtype=torch.uint8, device="cuda")
    plan.set_output("profile", 2)
    outs = []
    for st in (torch.cuda.default_stream(), torch.cuda.Stream()):
        out = torch.full((plan.out_offsets[-1],), 1e9, dtype=torch.float32, device="cuda")
        torch.cuda.synchronize()
        plan.run(x, out, ws, stream=st)
        plan.run(x, out, ws, stream=st)
        binding.scd_check_device(st)
        outs.append(out)
    assert torch.equal(outs[0], outs[1])
    plan.close()
