"""What the workspace's padding holds does not matter, in the adjoint and in
replays as in forward solves: rows and columns past the last 32-wide block are
never written and never reach a result.  A workspace filled with NaN in every
type gives the bits of a cleared one, with the S0 tape (its slices' padding) and
with FP32 checkpoints (copied, mirrored and split with their padding)."""

import pytest

from paper_2203_09621_gb300.workloads import make_instance

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2203_09621_gb300 import dmpt  # noqa: E402

DEV = torch.device("cuda:0")


@pytest.mark.parametrize("precision", ["dual_fp16", "dual_bf16"])
@pytest.mark.parametrize("n,k,cta_pair", [(33, 1, 1), (257, 2, 1), (700, 1, 1), (1030, 0, 1),
                                          (300, 1, 0)])
def test_adjoint_and_replay_on_a_filled_workspace(precision, n, k, cta_pair):
    ctx = dmpt.context(0)
    x = make_instance(f"pad{n}", n, n // 2, (-2.0, -0.1), (0.1, 2.0), seed=9650 + n, k=max(k, 1))
    H, H1 = torch.from_numpy(x.H).to(DEV), torch.from_numpy(x.H1).to(DEV)
    G = H1[0]
    kw = dict(cta_pair=cta_pair)

    def run(every, fill):
        nbytes = ctx.workspace_size(n, k, dmpt.options(precision=precision, ckpt_every=every, **kw))
        ws = torch.full((nbytes + 256,), fill, dtype=torch.uint8, device=DEV)
        P, P1, info = ctx.sp2_response(H, H1 if k else None, x.n_occ, precision=precision,
                                       ckpt_every=every, workspace=ws, **kw)
        assert info.converged
        out = [P, ctx.sp2_backward(G, ws, **kw)] + ([P1] if k else [])
        if every == 1 and k:
            out.append(ctx.response_replay(2.0 * H1, ws, precision=precision, **kw)[0])
        return out

    for every in (1, 4):
        for a, b in zip(run(every, 0), run(every, 0xFF)):
            assert torch.isfinite(a).all() and torch.equal(a, b)
