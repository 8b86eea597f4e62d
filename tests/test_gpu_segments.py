"""Ends of the recomputed segments in the checkpointed backward.

At each segment's end the step kernel between recompute layers hands the
control block to the decide step of the adjoint, which must read it only after
that kernel has finished: with an older copy the adjoint layers would run from
the wrong S0 state.  Short segments, many segment ends, every result equal to
the full tape's bit for bit.
"""

import pytest

from paper_2203_09621_gb300.workloads import make_instance

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2203_09621_gb300 import dmpt  # noqa: E402

DEV = torch.device("cuda:0")


@pytest.mark.parametrize("n,cta_pair", [(64, 1), (300, 1), (300, 0)])
@pytest.mark.parametrize("ckpt", [2, 3, 5])
def test_every_segment_end_sees_the_finished_recompute(n, cta_pair, ckpt):
    ctx = dmpt.context(0)
    x = make_instance(f"seg{n}", n, n // 2, (-2.0, -0.05), (0.05, 2.0), seed=9800 + n)
    H = torch.from_numpy(x.H).to(DEV)
    G = torch.from_numpy(x.H1[0]).to(DEV)

    def forward(every):
        opts = dmpt.options(ckpt_every=every, cta_pair=cta_pair)
        ws = torch.empty(ctx.workspace_size(n, 0, opts) + 256, dtype=torch.uint8, device=DEV)
        _, _, info = ctx.sp2_response(H, None, x.n_occ, ckpt_every=every, cta_pair=cta_pair,
                                      workspace=ws)
        assert info.converged and info.d0_layer > 2 * every   # three segments or more
        return ws

    full = ctx.sp2_backward(G, forward(1), cta_pair=cta_pair)
    ws = forward(ckpt)
    for _ in range(20):
        assert torch.equal(ctx.sp2_backward(G, ws, cta_pair=cta_pair), full)


# The tile width of a launch follows the jobs that run in it (forward: square
# and responses; recompute: the square; adjoint: one response; replay: the
# responses), so it differs between them; every width must give the bits of the
# single-CTA kernel, which has one width (K sweeps forwards in both).

def solve(ctx, x, k, n, every, **kw):
    H = torch.from_numpy(x.H).to(DEV)
    H1 = torch.from_numpy(x.H1[:k]).to(DEV) if k else None
    opts = dmpt.options(ckpt_every=every, **kw)
    ws = torch.empty(ctx.workspace_size(n, k, opts) + 256, dtype=torch.uint8, device=DEV)
    P, P1, info = ctx.sp2_response(H, H1, x.n_occ, ckpt_every=every, workspace=ws, **kw)
    assert info.converged
    return P, P1, ws


@pytest.mark.parametrize("n,k,ckpt", [(290, 0, 3), (1100, 0, 4), (1290, 2, 8), (2304, 1, 8),
                                      (2304, 0, 8)])
def test_widths_of_the_backward_give_the_same_bits(n, k, ckpt):
    ctx = dmpt.context(0)
    x = make_instance(f"wj{n}", n, n // 2, (-2.0, -0.1), (0.1, 2.0), seed=9750 + n, k=max(k, 1))
    G = torch.from_numpy(x.H1[0]).to(DEV)
    grads = []
    for every, kw in [(1, dict(k_snake=0)), (ckpt, dict(k_snake=0)), (1, dict(cta_pair=0))]:
        P, P1, ws = solve(ctx, x, k, n, every, **kw)
        grads.append((P, P1, ctx.sp2_backward(G, ws, **kw)))
    for P, P1, g in grads[1:]:
        assert torch.equal(P, grads[0][0]) and torch.equal(g, grads[0][2])
        assert k == 0 or torch.equal(P1, grads[0][1])


@pytest.mark.parametrize("n,k", [(300, 3), (700, 3), (1290, 1), (1536, 3)])
def test_widths_of_a_replay_give_the_same_bits(n, k):
    ctx = dmpt.context(0)
    x = make_instance(f"wr{n}", n, n // 2, (-2.0, -0.1), (0.1, 2.0), seed=9770 + n, k=k)
    H1 = torch.from_numpy(x.H1).to(DEV)
    outs = []
    for kw in (dict(k_snake=0), dict(cta_pair=0)):
        _, P1, ws = solve(ctx, x, k, n, 1, **kw)
        outs.append((P1, ctx.response_replay(H1, ws, **kw)[0]))
    for P1, P1r in outs:
        assert torch.equal(P1, outs[0][0]) and torch.equal(P1r, outs[0][1])
