"""Solves of several threads on one handle.

The shared context hands one handle to every thread; single solves with their
own workspace and stream run side by side on it, each following its own run,
and give the bits they give alone.  More threads than the handle has progress
words: the rest wait their turn.
"""

import threading

import pytest

from paper_2203_09621_gb300.workloads import make_instance

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2203_09621_gb300 import dmpt  # noqa: E402

DEV = torch.device("cuda:0")


def run_threads(jobs):
    errors = []

    def guarded(job):
        try:
            job()
        except BaseException as e:      # reported by the test's own thread
            errors.append(e)

    ts = [threading.Thread(target=guarded, args=(j,)) for j in jobs]
    for t in ts:
        t.start()
    for t in ts:
        t.join(timeout=120)
    assert not any(t.is_alive() for t in ts)
    if errors:
        raise errors[0]


@pytest.mark.parametrize("threads,repeats", [(4, 12), (80, 2)])
def test_single_solves_share_a_handle(threads, repeats):
    ctx = dmpt.context(0)
    kinds = [(130, 1, "dual_fp16"), (300, 2, "dual_bf16"), (96, 1, "fp64"), (200, 1, "fp32")]
    cases = []
    for n, k, prec in kinds:
        x = make_instance(f"t{n}", n, n // 2, (-2.0, -0.1), (0.1, 2.0), seed=9500 + n, k=k)
        H, H1 = torch.from_numpy(x.H).to(DEV), torch.from_numpy(x.H1).to(DEV)
        nbytes = ctx.workspace_size(n, k, dmpt.options(precision=prec))
        cases.append((H, H1, x.n_occ, prec, nbytes, ctx.sp2_response(H, H1, x.n_occ, precision=prec)))
    torch.cuda.synchronize()

    def job(i):
        H, H1, n_occ, prec, nbytes, (P, P1, ref) = cases[i % len(cases)]
        with torch.cuda.stream(torch.cuda.Stream()):
            ws = torch.empty(nbytes + 256, dtype=torch.uint8, device=DEV)
            for _ in range(repeats):
                Pt, P1t, info = ctx.sp2_response(H, H1, n_occ, precision=prec, workspace=ws)
                assert info.layers == ref.layers and info.converged
                assert torch.equal(Pt, P) and torch.equal(P1t, P1)

    run_threads([lambda i=i: job(i) for i in range(threads)])


def test_density_with_gradient_from_several_threads():
    n = 200
    x = make_instance("td", n, n // 2, (-2.0, -0.1), (0.1, 2.0), seed=9499)
    G = torch.from_numpy(x.H1[0]).to(DEV)

    def solve(out, i):
        with torch.cuda.stream(torch.cuda.Stream()):
            H = torch.from_numpy(x.H).to(DEV).requires_grad_(True)
            P = dmpt.density(H, x.n_occ)
            (g,) = torch.autograd.grad(P, H, G)
            out[i] = (P.detach().cpu(), g.cpu())

    ref = [None]
    solve(ref, 0)
    outs = [None] * 6
    run_threads([lambda i=i: solve(outs, i) for i in range(6)])
    for P, g in outs:
        assert torch.equal(P, ref[0][0]) and torch.equal(g, ref[0][1])
