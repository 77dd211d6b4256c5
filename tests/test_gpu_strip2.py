"""SSCA strips of a length N = N1 N2 with mixed-radix factors (mix2.cuh): even and odd factors, lengths of each
parity and remainder modulo 4, short and long tails of the tiles, and a length without such a split; auto, cross
and conjugate against the FP64 oracle.  Tolerance: the FP32 form's 1e-5 of max |S|."""
import numpy as np
import pytest

from oracle import scd_oracle as orc
from paper_2506_18003_gb300 import binding, signals

pytestmark = pytest.mark.gpu

FP32_TOL = 1e-5


@pytest.fixture(scope="module")
def torch():
    import torch as t
    assert t.cuda.is_available(), "GPU tests need CUDA"
    binding.load()
    return t


@pytest.mark.parametrize("N", [4116, 4374, 4410, 5000, 6561, 10000, 19683, 44100, 48000, 50001, 100000, 250000])
@pytest.mark.parametrize("variant", ["auto", "cross", "conjugate"])
def test_strips_match_oracle(torch, N, variant):
    Np = 64 if N < 50000 else 16
    x = signals.modulated("qpsk", N, 4, 0.1, 5.0, seed=6300 + N % 97)
    y = signals.modulated("bpsk", N, 8, -0.05, 5.0, seed=6301 + N % 97)
    a = np.random.default_rng(N).uniform(0.1, 1.0, Np).astype(np.float32)
    kw, okw = {}, {}
    if variant == "cross":
        kw, okw = {"y": torch.from_numpy(y).cuda()}, {"y": y}
    elif variant == "conjugate":
        kw, okw = {"conjugate": True}, {"conjugate": True}
    S = binding.scd_ssca(torch.from_numpy(x).cuda(), Np, window=torch.from_numpy(a).cuda(), **kw)
    binding.scd_check_device()
    B = binding.scd_ssca(torch.from_numpy(x).cuda(), Np, window=torch.from_numpy(a).cuda(), schedule="stages", **kw)
    assert (S - B).abs().max().item() / S.abs().max().item() <= FP32_TOL   # Bluestein's strips
    ch = np.array(sorted({0, 1, Np // 4, Np // 2 - 1, Np // 2, Np // 2 + 1, Np - 1}))
    ref = orc.ssca(x, a, Np, channels=ch, chunk=1 << 15, **okw)
    got = S[torch.from_numpy(ch).cuda()].cpu().numpy()
    assert float(np.max(np.abs(got - ref))) / S.abs().max().item() <= FP32_TOL
