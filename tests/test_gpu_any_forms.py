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


@pytest.mark.parametrize("P", [121, 143])
def test_fam_factors_without_a_radix(torch, P):
    """11 and 13 are no radices: products of them run by Bluestein's identity."""
    Np, L = 32, 8
    x = signals.modulated("qpsk", (P - 1) * L + Np, 4, 0.1, 5.0, seed=9500 + P)
    a = orc.hamming_window(Np)
    S = binding.scd_fam(torch.from_numpy(x).cuda(), Np, L, P)
    binding.scd_check_device()
    ref = orc.fam(x, a, Np, L, P)
    assert float(np.max(np.abs(S.cpu().numpy() - ref)) / np.max(np.abs(ref))) <= FP32_TOL


def test_ssca_factors_without_a_radix(torch):
    """12100 = 110 x 110: the default equals the explicit staged schedule, Bluestein's strips."""
    N, Np = 12100, 32
    x = torch.from_numpy(signals.modulated("qpsk", N, 4, 0.1, 5.0, seed=9600)).cuda()
    S = binding.scd_ssca(x, Np)
    assert torch.equal(S, binding.scd_ssca(x, Np, schedule="stages"))
    ch = np.array([0, 15, 16, 31])
    ref = orc.ssca(x.cpu().numpy(), orc.hamming_window(Np), Np, channels=ch)
    got = S[torch.from_numpy(ch).cuda()].cpu().numpy()
    assert float(np.max(np.abs(got - ref))) / S.abs().max().item() <= FP32_TOL
