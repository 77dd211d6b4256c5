"""FAM pair transforms of any P on the packed lanes (bluestein2.cuh): the smallest and largest P of every
cyclic length 64 .. 4096 (17 and 2047 at the ends), auto, cross and conjugate, against the FP64
oracle.  Tolerance: the FP32 form's 1e-5 of max |S|."""
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


@pytest.mark.parametrize("P", [17, 31, 33, 63, 65, 127, 129, 255, 257, 511, 513, 1000, 1023, 1025, 2047])
@pytest.mark.parametrize("variant", ["auto", "cross", "conjugate"])
def test_pairs_match_oracle(torch, P, variant):
    Np, L = (16, 3) if P % 4 == 1 else (32, 5)
    N = (P - 1) * L + Np
    x = signals.modulated("qpsk", N, 4, 0.1, 5.0, seed=4300 + P)
    y = signals.modulated("bpsk", N, 8, -0.05, 5.0, seed=4301 + P)
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
