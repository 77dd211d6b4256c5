"""Normalised SSCA estimates of very large and very small samples: the lag products are formed before the window,
so the normalisation must reach them before their squares leave the range of a float.  The estimate does
not change with the samples' scale: a power of two gives the same bits."""
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


@pytest.mark.parametrize("N,Np", [(1 << 12, 16), (1 << 14, 64), (1 << 17, 256)])
@pytest.mark.parametrize("mode", ["power", "peak"])
def test_scale_does_not_matter(torch, N, Np, mode):
    x = signals.modulated("qpsk", N, 4, 0.1, 5.0, seed=8300 + Np)
    a = np.random.default_rng(Np).uniform(0.1, 1.0, Np).astype(np.float32)
    xd, ad = torch.from_numpy(x).cuda(), torch.from_numpy(a).cuda()
    base = binding.scd_ssca(xd, Np, window=ad, normalise=mode)
    binding.scd_check_device()
    ch = np.array(sorted({0, Np // 4, Np // 2, Np - 1}))
    ref = orc.ssca(x, a, Np, channels=ch, chunk=1 << 15, normalise=binding.NORMALISE[mode])
    got = base[torch.from_numpy(ch).cuda()].cpu().numpy()
    assert float(np.max(np.abs(got - ref))) / base.abs().max().item() <= FP32_TOL
    for e in (-62, -20, 20, 62):
        S = binding.scd_ssca(xd * 2.0 ** e, Np, window=ad, normalise=mode)
        assert torch.equal(S, base), e
    T = binding.scd_ssca(xd * 2.0 ** 55, Np, window=ad, normalise=mode, schedule="stages")
    assert (T - base).abs().max().item() / base.abs().max().item() <= FP32_TOL
