"""FP32 <-> FP64 conversions of the element-wise kernels: scaling the inputs of a
linear map by a power of two scales its result exactly, far from 1 as well
(inputs around 2^-40 and 2^40, outputs of both signs and
the complement form), and an output never differs from its mirror element.
"""

import pytest

from paper_2203_09621_gb300.workloads import make_instance

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2203_09621_gb300 import dmpt  # noqa: E402

DEV = torch.device("cuda:0")


def instance(n, n_occ):
    x = make_instance(f"c{n}", n, n_occ, (-2.0, -0.1), (0.1, 2.0), seed=9900 + n)
    return torch.from_numpy(x.H).to(DEV), torch.from_numpy(x.H1).to(DEV)


@pytest.mark.parametrize("n,n_occ", [(70, 35), (300, 220)])
@pytest.mark.parametrize("exponent", [-40, -7, 5, 40])
def test_response_scales_exactly(n, n_occ, exponent):
    ctx = dmpt.context(0)
    H, H1 = instance(n, n_occ)
    P, P1, _ = ctx.sp2_response(H, H1, n_occ)
    Ps, P1s, _ = ctx.sp2_response(H, H1 * 2.0 ** exponent, n_occ)
    torch.cuda.synchronize()
    assert torch.equal(P, Ps) and torch.equal(P1s, P1 * 2.0 ** exponent)


@pytest.mark.parametrize("n", [70, 300])
@pytest.mark.parametrize("exponent", [-40, 40])
def test_adjoint_scales_exactly(n, exponent):
    ctx = dmpt.context(0)
    H, H1 = instance(n, n // 2)
    opts = dmpt.options(ckpt_every=1)
    ws = torch.empty(ctx.workspace_size(n, 0, opts) + 256, dtype=torch.uint8, device=DEV)
    ctx.sp2_response(H, None, n // 2, ckpt_every=1, workspace=ws)
    G = torch.randn(n, n, dtype=torch.float64, device=DEV, generator=torch.Generator(DEV).manual_seed(3))
    g = ctx.sp2_backward(G, ws).clone()
    gs = ctx.sp2_backward(G * 2.0 ** exponent, ws)
    torch.cuda.synchronize()
    assert torch.equal(gs, g * 2.0 ** exponent)
    assert torch.equal(g, g.T)
