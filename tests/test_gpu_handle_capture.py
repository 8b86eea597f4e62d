"""A handle may be created and destroyed while a stream capture is under way:
neither is part of the captured work, and neither ends the capture."""

import pytest

from paper_2203_09621_gb300.workloads import make_workload

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2203_09621_gb300 import dmpt  # noqa: E402


def test_handle_created_and_destroyed_during_a_capture():
    x = torch.arange(8, device="cuda:0", dtype=torch.float64)
    y = torch.zeros_like(x)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        ctx = dmpt.Context(0)
        y.copy_(x + 1)
        dmpt.Context(0).close()
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(y, x + 1)
    inst = make_workload(1)
    H, H1 = (torch.from_numpy(a).to("cuda:0") for a in (inst.H, inst.H1))
    P, P1, info = ctx.sp2_response(H, H1, inst.n_occ)
    Pr, P1r, _ = dmpt.context(0).sp2_response(H, H1, inst.n_occ)
    assert info.converged and torch.equal(P, Pr) and torch.equal(P1, P1r)
