"""FAM lengths without a mixed-radix plan at the cyclic lengths 4096 and 8192, on both sides of the rules that choose
between the one-pair kernels (uncapped, two blocks per SM) and the packed one: fewer and more pairs than SMs,
short and full last rounds; auto and cross, sampled pairs against the FP64 oracle.  Tolerance: the FP32
form's 1e-5 of max |S|."""
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


@pytest.mark.parametrize("Np", [16, 32, 64])
@pytest.mark.parametrize("P", [1025, 2039, 2053, 4091])
@pytest.mark.parametrize("variant", ["auto", "cross"])
def test_forms_match_oracle(torch, Np, P, variant):
    L = max(1, Np // 8)
    N = (P - 1) * L + Np
    x = signals.modulated("qpsk", N, 4, 0.1, 5.0, seed=9300 + Np + P)
    y = signals.modulated("bpsk", N, 8, -0.05, 5.0, seed=9301 + Np + P)
    a = np.random.default_rng(P).uniform(0.1, 1.0, Np).astype(np.float32)
    kw, okw = ({"y": torch.from_numpy(y).cuda()}, {"y": y}) if variant == "cross" else ({}, {})
    S = binding.scd_fam(torch.from_numpy(x).cuda(), Np, L, P, window=torch.from_numpy(a).cuda(), **kw)
    binding.scd_check_device()
    g = np.random.default_rng(7)
    kh = np.concatenate([[0, Np - 1, 0, Np - 1], g.integers(0, Np, 40)])
    lh = np.concatenate([[0, Np - 1, Np - 1, 0], g.integers(0, Np, 40)])
    ref = orc.fam_pairs(x, a, Np, L, P, kh, lh, **okw)
    got = S[torch.from_numpy(kh).cuda(), torch.from_numpy(lh).cuda()].cpu().numpy()
    assert float(np.max(np.abs(got - ref))) / S.abs().max().item() <= FP32_TOL
