"""FAM pair transforms on the packed lanes (P = 32, 512 and the auto estimate at 1024; fam2.cuh): every
cell against the FP64 oracle for every channel count, auto, cross and conjugate, through scd_fam; batch
plans at those sizes and their neighbours against the oracle and, within the tolerance, the staged
kernels.  Tolerance: the FP32 form's 1e-5 of max |S|."""
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


@pytest.mark.parametrize("P", [32, 512, 1024])
@pytest.mark.parametrize("Np", [16, 64, 256])
@pytest.mark.parametrize("variant", ["auto", "cross", "conjugate"])
def test_pairs_match_oracle(torch, Np, P, variant):
    L = 3
    N = (P - 1) * L + Np
    x = signals.modulated("qpsk", N, 4, 0.1, 5.0, seed=3300 + Np + P)
    y = signals.modulated("bpsk", N, 8, -0.05, 5.0, seed=3301 + Np + P)
    a = np.random.default_rng(P).uniform(0.1, 1.0, Np).astype(np.float32)
    kw, okw = {}, {}
    if variant == "cross":
        kw, okw = {"y": torch.from_numpy(y).cuda()}, {"y": y}
    elif variant == "conjugate":
        kw, okw = {"conjugate": True}, {"conjugate": True}
    S = binding.scd_fam(torch.from_numpy(x).cuda(), Np, L, P, window=torch.from_numpy(a).cuda(), **kw)
    binding.scd_check_device()
    g = np.random.default_rng(7)
    kh = np.concatenate([np.arange(Np), g.integers(0, Np, 4 * Np)])       # the diagonal and random pairs
    lh = np.concatenate([np.arange(Np), g.integers(0, Np, 4 * Np)])
    ref = orc.fam_pairs(x, a, Np, L, P, kh, lh, **okw)
    got = S[torch.from_numpy(kh).cuda(), torch.from_numpy(lh).cuda()].cpu().numpy()
    assert float(np.max(np.abs(got - ref))) / S.abs().max().item() <= FP32_TOL
    if variant == "auto":                                                 # mirrored rows: exact conjugates
        q = torch.arange(P, device="cuda")
        off = ~torch.eye(Np, dtype=torch.bool, device="cuda")             # (a diagonal row is its own transform)
        mirrored = S.transpose(0, 1)[:, :, (P - q) % P].conj().resolve_conj()
        assert torch.equal(S[off], mirrored[off])


@pytest.mark.parametrize("Np,L", [(16, 4), (64, 16)])
def test_batch_default_schedule(torch, Np, L):
    lengths = [P * L + Np for P in (32, 33, 64, 511, 512, 600, 1024, 1025, 2048)]
    sigs = [signals.batch_signal(1300 + i, n) for i, n in enumerate(lengths)]
    plan = binding.BatchPlan("fam", lengths, Np, L)
    x = torch.from_numpy(np.concatenate(sigs)).cuda()
    ws = torch.empty(plan.workspace_bytes, dtype=torch.uint8, device="cuda")
    outs = []
    for sched in ("auto", "stages"):
        plan.set_schedule(sched)
        out = torch.empty(plan.out_offsets[-1], dtype=torch.complex64, device="cuda")
        plan.run(x, out, ws)
        binding.scd_check_device()
        outs.append(out)
    a = orc.hamming_window(Np)
    for i, s in enumerate(sigs):
        ref = orc.fam(s, a, Np, L, plan.sizes[i])
        m = np.max(np.abs(ref))
        assert np.max(np.abs(plan.output(outs[0], i).cpu().numpy() - ref)) / m <= FP32_TOL, i
        assert (plan.output(outs[0], i) - plan.output(outs[1], i)).abs().max().item() / m <= FP32_TOL, i
    plan.close()
