"""SSCA lengths that are not powers of two, taken in turn: the split of a length is not searched again on every
call, the estimates stay those of the lengths taken alone, and more lengths than are kept do no harm."""
import time

import pytest

from paper_2506_18003_gb300 import binding

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    import torch as t
    assert t.cuda.is_available(), "GPU tests need CUDA"
    binding.load()
    return t


def _state(torch, N, Np):
    return (torch.randn(N, dtype=torch.complex64, device="cuda"), torch.empty((Np, N), dtype=torch.complex64, device="cuda"),
            torch.empty(binding.load().scd_ssca_workspace_bytes(N, Np, 0), dtype=torch.uint8, device="cuda"))


def _host_us(torch, states, Np):
    """Host time of a call, the least of several rounds of 40 (few enough to fit the launch queue)."""
    best = 1e9
    for _ in range(12):
        torch.cuda.synchronize()
        t = time.perf_counter()
        for i in range(40):
            x, out, ws = states[i % len(states)]
            binding.scd_ssca(x, Np, out=out, workspace=ws)
        best = min(best, (time.perf_counter() - t) / 40 * 1e6)
    return best


def test_two_lengths_in_turn(torch):
    Np = 16
    a, b = _state(torch, 44100, Np), _state(torch, 48000, Np)
    for x, out, ws in (a, b):                                # tables
        binding.scd_ssca(x, Np, out=out, workspace=ws)
    want = [a[1].clone(), b[1].clone()]
    alone = max(_host_us(torch, [a], Np), _host_us(torch, [b], Np))
    assert _host_us(torch, [a, b], Np) <= 1.5 * alone        # the search alone takes more than a call does
    binding.scd_check_device()
    assert torch.equal(a[1], want[0]) and torch.equal(b[1], want[1])


def test_many_lengths(torch):
    Np, lengths = 16, [4100 + 4 * i for i in range(80)]
    first = {}
    for turn in range(2):
        for N in lengths:
            x = torch.arange(N, device="cuda").to(torch.complex64) * 1j
            S = binding.scd_ssca(x, Np)
            if turn == 0:
                first[N] = S
            else:
                assert torch.equal(S, first[N]), N
    binding.scd_check_device()
