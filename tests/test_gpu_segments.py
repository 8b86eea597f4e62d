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
