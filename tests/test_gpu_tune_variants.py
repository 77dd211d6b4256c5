"""scd_ssca_tune keeps the auto estimate's choice apart from the cross and conjugate estimates', whose kernels
differ: tuning one of those, or a cache file that holds such a choice, leaves the auto estimates on the
lag-domain kernels.  Each case runs in a process of its own (the choices are kept per process)."""
import json
import os
import subprocess
import sys

import pytest

from paper_2506_18003_gb300 import binding

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
HEAD = """
import ctypes, sys, torch
from paper_2506_18003_gb300 import binding
lib = binding.load()
N, Np, variant = int(sys.argv[1]), int(sys.argv[2]), sys.argv[3]
x = torch.randn(N, dtype=torch.complex64, device="cuda")
def launches(**kw):
    n = lib.scd_launch_count()
    binding.scd_ssca(x, Np, **kw)
    return lib.scd_launch_count() - n
"""
TUNE = """
out = torch.empty((Np, N), dtype=torch.complex64, device="cuda")
ws = torch.empty(lib.scd_ssca_workspace_bytes(N, Np, 0), dtype=torch.uint8, device="cuda")
want = binding.scd_ssca(x, Np)
o = binding.make_opts(workspace=ws, y=x if variant == "cross" else None, conjugate=variant == "conjugate")
binding.check(lib.scd_ssca_tune(x.data_ptr(), N, Np, None, out.data_ptr(), ctypes.byref(o), 1), "tune")
if variant != "auto":
    assert torch.equal(binding.scd_ssca(x, Np), want)          # the same kernels as before
binding.scd_check_device()
"""


def _run(code, cache, N, Np, variant):
    r = subprocess.run([sys.executable, "-c", HEAD + code, str(N), str(Np), variant], cwd=ROOT, capture_output=True,
                       env=dict(os.environ, SCD_TUNE_CACHE=str(cache)), text=True, timeout=300)
    assert r.returncode == 0, r.stderr
    return r.stdout


@pytest.mark.parametrize("variant", ["auto", "cross", "conjugate"])
@pytest.mark.parametrize("N,Np", [(1 << 13, 128), (1 << 14, 16)])   # FUSED's tiles fit; do not fit
def test_tuning_a_variant_leaves_auto_alone(tmp_path, variant, N, Np):
    assert binding.load()
    cache = tmp_path / "tune.json"
    _run(TUNE, cache, N, Np, variant)
    keys = {e["key"].split("|", 1)[1] for e in json.load(open(cache))["entries"]}
    size = f"|N={N}|Np={Np}|p=0"
    assert keys == ({"ssca" + size, "ssca-lag" + size} if variant == "auto" else {"ssca" + size})


def test_cache_file_of_the_other_kernels(tmp_path):
    """A file that says PERSISTENT (one launch) and was never timed against the lag domain (three)."""
    import torch
    N, Np = 1 << 15, 32
    cache = tmp_path / "tune.json"
    code = "print(launches(), launches(y=x)); binding.scd_check_device()"
    assert _run(code, cache, N, Np, "").split() == ["3", "3"]
    p = torch.cuda.get_device_properties(0)
    key = f"{p.name}/sm{10 * p.major + p.minor}|ssca|N={N}|Np={Np}|p=0"
    cache.write_text('{"scd_tune_version": 1, "entries": [\n'
                     f'{{"key": "{key}", "schedule": 2, "item_kib": 128, "slot_kib": 16384, "ms": 0.1}}\n]}}\n')
    assert _run(code, cache, N, Np, "").split() == ["3", "1"]  # the cross estimate follows it, the auto one does not
