"""Mixed-radix FAM pair transforms (mix2.cuh): lengths that use every radix 2 .. 16 first, in the middle and
last, of two, three and four passes, up to the largest size, and products the plan refuses (17 times a
factor, above 4096); auto, cross and conjugate against the FP64 oracle.  Tolerance: the FP32 form's 1e-5
of max |S|."""
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


@pytest.mark.parametrize("P", [18, 20, 21, 25, 34, 48, 49, 63, 75, 96, 98, 100, 105, 200, 225, 240, 243, 336, 343, 500,
                               686, 810, 1000, 1125, 1536, 2187, 2401, 3000, 3840, 4050, 4095, 4116])
@pytest.mark.parametrize("variant", ["auto", "cross", "conjugate"])
def test_pairs_match_oracle(torch, P, variant):
    Np, L = (64, 16) if P < 120 else (16, 4)                   # several tiles of many units; tiles of few
    N = (P - 1) * L + Np
    x = signals.modulated("qpsk", N, 4, 0.1, 5.0, seed=5300 + P)
    y = signals.modulated("bpsk", N, 8, -0.05, 5.0, seed=5301 + P)
    a = np.random.default_rng(P).uniform(0.1, 1.0, Np).astype(np.float32)
    kw, okw = {}, {}
    if variant == "cross":
        kw, okw = {"y": torch.from_numpy(y).cuda()}, {"y": y}
    elif variant == "conjugate":
        kw, okw = {"conjugate": True}, {"conjugate": True}
    S = binding.scd_fam(torch.from_numpy(x).cuda(), Np, L, P, window=torch.from_numpy(a).cuda(), **kw)
    binding.scd_check_device()
    kh, lh = np.divmod(np.arange(Np * Np), Np)
    ref = orc.fam_pairs(x, a, Np, L, P, kh, lh, **okw).reshape(Np, Np, P)
    assert float(np.max(np.abs(S.cpu().numpy() - ref))) / float(np.max(np.abs(ref))) <= FP32_TOL
