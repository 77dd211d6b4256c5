"""SSCA auto estimates in the lag domain (what AUTO runs for powers of two in the FP32 form): the
identity itself in FP64 on the CPU, and the kernels against the FP64 oracle at every strip split
(N = 2^12 .. 2^20), every channel count, through scd_ssca and through batch plans, with the
profiles of each.  Tolerance: the FP32 form's 1e-5 of max |S|."""
import numpy as np
import pytest

from oracle import scd_oracle as orc
from paper_2506_18003_gb300 import binding, signals

FP32_TOL = 1e-5


def _lag_domain(x, a, Np):
    """S from the transforms of the lag products of the lags m >= 0 alone, complex128."""
    N, H = len(x), Np // 2
    x = x.astype(np.complex128)
    c = np.arange(N)
    S = np.zeros((Np, N), dtype=np.complex128)
    R = [np.fft.fft(np.concatenate([x[m:] * np.conj(x[:N - m]), np.zeros(m)])) for m in range(H + 1)]
    for kh in range(Np):
        k = kh - H
        v = np.zeros(N, dtype=np.complex128)
        for m in range(-H, H):
            r = R[m] if m >= 0 else orc.twiddle(N, -c * m) * np.conj(R[-m][(-c) % N])
            v += float(a[m + H]) * orc.twiddle(Np, k * m) * r
        S[kh, (c - k * (N // Np) + N // 2) % N] = v
    return S


@pytest.mark.parametrize("N,Np", [(64, 16), (128, 32), (256, 16)])
def test_lag_identity(N, Np):
    g = np.random.default_rng(5)
    x = (g.standard_normal(N) + 1j * g.standard_normal(N)).astype(np.complex64)
    a = g.uniform(0.1, 1.0, Np).astype(np.float32)             # no symmetry to lean on
    ref = orc.ssca(x, a, Np)
    assert np.max(np.abs(_lag_domain(x, a, Np) - ref)) / np.max(np.abs(ref)) <= 1e-12


@pytest.fixture(scope="module")
def torch():
    import torch as t
    assert t.cuda.is_available(), "GPU tests need CUDA"
    binding.load()
    return t


def _err(torch, S, x, a, Np):
    ch = np.array(sorted({0, 1, Np // 4, Np // 2 - 1, Np // 2, Np // 2 + 1, Np - 1}))
    ref = orc.ssca(x, a, Np, channels=ch, chunk=1 << 15)
    got = S[torch.from_numpy(ch).cuda()].cpu().numpy()
    return float(np.max(np.abs(got - ref))) / S.abs().max().item()


@pytest.mark.gpu
@pytest.mark.parametrize("e", range(12, 21))
@pytest.mark.parametrize("Np", [16, 32, 64, 128, 256])
def test_lag_matches_oracle(torch, e, Np):
    N = 1 << e
    x = signals.modulated("qpsk", N, 4, 0.1, 5.0, seed=3100 + Np + e)
    a = np.random.default_rng(e).uniform(0.1, 1.0, Np).astype(np.float32)
    arena = torch.from_numpy(np.concatenate([np.zeros(1, np.complex64), x])).cuda()
    S = binding.scd_ssca(arena[1:], Np, window=torch.from_numpy(a).cuda())   # 8-byte aligned input
    binding.scd_check_device()
    assert _err(torch, S, x, a, Np) <= FP32_TOL
    if N * Np <= 1 << 23:                                      # every cell against the staged kernels
        T = binding.scd_ssca(arena[1:], Np, window=torch.from_numpy(a).cuda(), schedule="stages")
        assert (S - T).abs().max().item() / T.abs().max().item() <= FP32_TOL
    del S, arena
    torch.cuda.empty_cache()


@pytest.mark.gpu
@pytest.mark.parametrize("Np", [16, 32, 256])
def test_lag_batch_and_profiles(torch, Np):
    """Batch plans at the channel counts and sizes the fused tiles do not take: estimates against
    the oracle and bit for bit against scd_ssca, profiles bit for bit against their estimates'."""
    lengths = [4097, 9000, 5000, 40001, 16384, 1 << 19]
    sigs = [signals.batch_signal(1200 + i, n) for i, n in enumerate(lengths)]
    x = torch.from_numpy(np.concatenate(sigs)).cuda()
    plan = binding.BatchPlan("ssca", lengths, Np)
    ws = torch.empty(plan.workspace_bytes, dtype=torch.uint8, device="cuda")
    out = torch.empty(plan.out_offsets[-1], dtype=torch.complex64, device="cuda")
    plan.run(x, out, ws)
    a = orc.hamming_window(Np)
    est = [plan.output(out, i) for i in range(len(lengths))]
    for i, s in enumerate(sigs):
        N = plan.sizes[i]
        assert _err(torch, est[i], s[:N].copy(), a, Np) <= FP32_TOL, i
        assert torch.equal(est[i], binding.scd_ssca(torch.from_numpy(s[:N].copy()).cuda(), Np)), i
    for power in (1, 2):
        plan.set_output("profile", power)
        prof = torch.empty(plan.out_offsets[-1], dtype=torch.float32, device="cuda")
        plan.run(x, prof, torch.empty(plan.workspace_bytes, dtype=torch.uint8, device="cuda"))
        binding.scd_check_device()
        for i in range(len(lengths)):
            same = binding.scd_ssca_alpha_profile(est[i], plan.sizes[i], Np, power=power)
            assert torch.equal(plan.output(prof, i), same), (i, power)
    plan.close()


@pytest.mark.gpu
def test_lag_capture_after_prepare(torch):
    """scd_prepare builds every table the default schedule needs: the call can be captured."""
    N, Np = 1 << 13, 64
    x = torch.randn(N, dtype=torch.complex64, device="cuda")
    binding.scd_prepare("ssca", N, Np)
    out = torch.empty((Np, N), dtype=torch.complex64, device="cuda")
    ws = torch.empty(binding.load().scd_ssca_workspace_bytes(N, Np, 0), dtype=torch.uint8, device="cuda")
    want = binding.scd_ssca(x, Np).clone()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        binding.scd_ssca(x, Np, out=out, workspace=ws)
    out.zero_()
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(out, want)
