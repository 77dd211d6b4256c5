"""SSCA estimates whose samples or window lie in the output's own memory (a receive buffer that the estimate
overwrites): the same as from separate buffers, under every schedule.  Tolerance: the FP32 form's 1e-5 of
max |S|."""
import pytest

from paper_2506_18003_gb300 import binding

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    import torch as t
    assert t.cuda.is_available(), "GPU tests need CUDA"
    binding.load()
    return t


@pytest.mark.parametrize("N,Np", [(1 << 12, 64), (1 << 13, 16), (1 << 16, 256), (5000, 32), (10007, 16)])
@pytest.mark.parametrize("at", ["first", "odd", "last"])
@pytest.mark.parametrize("schedule", ["auto", "fused", "stages"])
def test_samples_inside_the_output(torch, N, Np, at, schedule):
    x = torch.randn(N, dtype=torch.complex64, device="cuda")
    want = binding.scd_ssca(x, Np, schedule="stages")
    out = torch.empty((Np, N), dtype=torch.complex64, device="cuda")
    o = {"first": 0, "odd": 3 * N + 1, "last": (Np - 1) * N}[at]
    inside = out.view(-1)[o:o + N]
    inside.copy_(x)
    binding.scd_ssca(inside, Np, out=out, schedule=schedule)
    binding.scd_check_device()
    assert (out - want).abs().max().item() / want.abs().max().item() <= 1e-5


@pytest.mark.parametrize("N,Np", [(1 << 12, 64), (1 << 13, 16)])
def test_window_inside_the_output(torch, N, Np):
    x = torch.randn(N, dtype=torch.complex64, device="cuda")
    a = torch.rand(Np, device="cuda") + 0.1
    want = binding.scd_ssca(x, Np, window=a, schedule="stages")
    out = torch.empty((Np, N), dtype=torch.complex64, device="cuda")
    inside = torch.view_as_real(out).view(-1)[2 * N + 8:2 * N + 8 + Np]
    inside.copy_(a)
    binding.scd_ssca(x, Np, window=inside, out=out)
    binding.scd_check_device()
    assert (out - want).abs().max().item() / want.abs().max().item() <= 1e-5
