"""Estimates queued back to back on one stream through one workspace, their inputs in turn, without a
synchronisation in between: dependent launches overlap the set-up of consecutive kernels, and every result
must still be the isolated call's, bit for bit (the pair and strip kernels read what the kernel before
them wrote to the same addresses as in the call before)."""
import pytest

from paper_2506_18003_gb300 import binding

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    import torch as t
    assert t.cuda.is_available(), "GPU tests need CUDA"
    binding.load()
    return t


def _queue(torch, call, xs, ws, calls):
    """call(x, out, workspace) for the inputs in turn; each result against the isolated call's."""
    want = []
    for x in xs:
        w = call(x, None, None)
        torch.cuda.synchronize()
        want.append(w)
    assert not torch.equal(want[0], want[1])
    outs = [torch.zeros_like(want[0]) for _ in range(calls)]
    torch.cuda.synchronize()
    for i, o in enumerate(outs):
        call(xs[i % len(xs)], o, ws)
    binding.scd_check_device()
    for i, o in enumerate(outs):
        assert torch.equal(o, want[i % len(xs)]), i


# scalar pair kernel, packed lanes, Bluestein on the packed lanes (37, 121: 11 is not a radix), mixed radices
@pytest.mark.parametrize("P", [8, 32, 37, 100, 121, 128, 1000, 1024, 2048])
@pytest.mark.parametrize("cross", [False, True])
def test_fam(torch, P, cross):
    Np, L = (64, 16) if P <= 1024 else (32, 8)
    N = (P - 1) * L + Np
    xs = [torch.randn(N, dtype=torch.complex64, device="cuda") for _ in range(3)]
    y = torch.randn(N, dtype=torch.complex64, device="cuda") if cross else None
    ws = torch.empty(binding.load().scd_fam_workspace_bytes(N, Np, L, P, 0), dtype=torch.uint8, device="cuda")
    _queue(torch, lambda x, o, w: binding.scd_fam(x, Np, L, P, out=o, workspace=w, y=y), xs, ws, 24)


@pytest.mark.parametrize("N", [1 << 12, 1 << 16, 5000, 44100])
def test_ssca(torch, N):
    Np = 64
    xs = [torch.randn(N, dtype=torch.complex64, device="cuda") for _ in range(3)]
    ws = torch.empty(binding.load().scd_ssca_workspace_bytes(N, Np, 0), dtype=torch.uint8, device="cuda")
    _queue(torch, lambda x, o, w: binding.scd_ssca(x, Np, out=o, workspace=w), xs, ws, 16)
