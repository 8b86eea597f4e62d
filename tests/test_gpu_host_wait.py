"""How the host waits for a running solve: it does not hold a core through long
layers, and it follows the device's schedule flags (yield, blocking), with the
same results."""

import os
import subprocess
import sys
import time

import pytest

from paper_2203_09621_gb300.workloads import make_instance

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2203_09621_gb300 import dmpt  # noqa: E402

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_long_layers_leave_the_core_to_others():
    """FP64 layers of about 20 ms: the calling thread sleeps most of the time."""
    n = 1900
    x = make_instance("hw", n, n // 2, (-2.0, -0.1), (0.1, 2.0), seed=9490)
    ctx = dmpt.context(0)
    H, H1 = (torch.from_numpy(a).to("cuda:0") for a in (x.H, x.H1))
    torch.cuda.synchronize()
    wall, cpu = time.perf_counter(), time.thread_time()
    _, _, info = ctx.sp2_response(H, H1, x.n_occ, precision="fp64")
    wall, cpu = time.perf_counter() - wall, time.thread_time() - cpu
    assert info.converged and wall > 0.2
    assert cpu < 0.6 * wall, (cpu, wall)


CHILD = """
import ctypes, sys
import torch
rt = ctypes.CDLL("libcudart.so.13")          # the one torch has loaded
assert rt.cudaSetDeviceFlags(int(sys.argv[1])) == 0
from paper_2203_09621_gb300 import dmpt
from paper_2203_09621_gb300.workloads import make_instance
f = ctypes.c_uint()
torch.zeros(1, device="cuda:0")
assert rt.cudaGetDeviceFlags(ctypes.byref(f)) == 0 and f.value & 7 == int(sys.argv[1]), f.value
x = make_instance("hf", 300, 150, (-2.0, -0.1), (0.1, 2.0), seed=9491)
H, H1 = (torch.from_numpy(a).to("cuda:0") for a in (x.H, x.H1))
ctx = dmpt.context(0)
outs = [ctx.sp2_response(H, H1, 150, **kw) for kw in ({}, dict(sync_every=1), dict(max_layers=3, raise_on_error=False))]
Ps, P1s, infos = ctx.sp2_response_batch([H, H], [H1, H1], [150, 150])
torch.cuda.synchronize()
assert outs[0][2].converged and outs[2][2].layers == 3
assert torch.equal(outs[0][1], outs[1][1]) and torch.equal(outs[0][1], P1s[1])
torch.save(outs[0][1].cpu(), sys.argv[2])
"""


def test_schedule_flags_give_the_same_results(tmp_path):
    results = []
    for flag in (0, 1, 2, 4):           # auto, spin, yield, blocking
        out = tmp_path / f"p1_{flag}.pt"
        env = dict(os.environ, PYTHONPATH=ROOT)
        subprocess.run([sys.executable, "-c", CHILD, str(flag), str(out)], check=True, cwd=ROOT,
                       env=env, timeout=300)
        results.append(torch.load(out))
    assert all(torch.equal(r, results[0]) for r in results)


def test_sync_every_sets_how_far_the_host_runs_ahead():
    """Layers of about 1 ms: the number issued beyond the last one that ran says
    how long the queue was.  Results do not depend on it."""
    n = 700
    x = make_instance("ha", n, n // 2, (-2.0, -0.1), (0.1, 2.0), seed=9492)
    ctx = dmpt.context(0)
    H, H1 = (torch.from_numpy(a).to("cuda:0") for a in (x.H, x.H1))
    P, P1, ref = ctx.sp2_response(H, H1, x.n_occ, precision="fp64")
    for sync_every in (1, 2, 3, 5, 16, 100):
        Ps, P1s, info = ctx.sp2_response(H, H1, x.n_occ, precision="fp64", sync_every=sync_every)
        assert info.layers == ref.layers and torch.equal(Ps, P) and torch.equal(P1s, P1)
        beyond = info.product_launches - info.layers
        # two layers ahead leave one beyond the last; a host that loses its core for
        # a few layers shortens a longer queue by as many
        if sync_every <= 4:
            assert 0 <= beyond <= 1
        elif sync_every == 5:
            assert beyond <= 5
        else:
            assert 2 <= beyond <= sync_every or info.product_launches == 100
