"""The conversions between FP32 and FP64 of the initial layer, the outputs and
the adjoint start, bit for bit against casts: rounding to nearest even (ties,
carries into the exponent), both ends of the normal range, subnormal results,
overflow, infinities and NaN.

H is diagonal with levels 0 and 1, so S_0 is the projector itself and every
layer returns a perturbation that couples occupied with empty levels unchanged:
P1 = -(H1 rounded to FP32) exactly.  The S0 recursion ends at its first layer
without an update, so dL/dH = -((G + G^T) / 2 rounded to FP32).
"""

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2203_09621_gb300 import dmpt  # noqa: E402

DEV = torch.device("cuda:0")
F64 = torch.float64


def mantissas():
    t = 2.0 ** -24                      # half a unit in the last place of FP32 at 1
    e = 2.0 ** -52
    return [1.0, 1 + t, 1 + t - e, 1 + t + e, 1 + 2 * t, 1 + 3 * t, 1 + 3 * t - e, 1 + 3 * t + e,
            1 + 5 * t, 1.5, 2 - 2 * t, 2 - t - e, 2 - t, 2 - t + e, 2 - t / 2, 2 - e]


def values(count, top, seed):
    """`count` doubles over the FP32 range and below it, both signs."""
    v = torch.tensor([m * 2.0 ** p for p in range(-153, top + 1) for m in mantissas()]
                     + [0.0, 2.0 ** -400, 2.0 ** -1050], dtype=F64)
    g = torch.Generator().manual_seed(seed)
    assert v.numel() < count
    r = (1 + torch.rand(count - v.numel(), generator=g, dtype=F64)) * torch.exp2(
        torch.randint(-153, top, (count - v.numel(),), generator=g).to(F64))
    v = torch.cat([v, r])[torch.randperm(count, generator=g)]
    return v * (torch.randint(0, 2, (count,), generator=g) * 2 - 1)


def levels(n, n_occ):
    H = torch.zeros(n, n, dtype=F64, device=DEV)
    H.diagonal()[n_occ:] = 1.0
    return H


@pytest.mark.parametrize("n,n_occ", [(256, 128), (301, 150), (256, 160)])   # the last: complement
def test_response_inputs_and_outputs_are_rounded_once(n, n_occ):
    H1 = torch.zeros(n, n, dtype=F64)
    # up to 2^126: the layer forms 2 S - S
    H1[:n_occ, n_occ:] = values(n_occ * (n - n_occ), 125, n).reshape(n_occ, n - n_occ)
    H1 = (H1 + H1.T).to(DEV)
    P, P1, info = dmpt.context(0).sp2_response(levels(n, n_occ), H1, n_occ, precision="fp32")
    assert info.converged and info.d0_layer == 1
    assert torch.equal(P, torch.eye(n, dtype=F64, device=DEV) - levels(n, n_occ))
    assert torch.equal(P1[0], -H1.to(torch.float32).to(F64))


def adjoint(n, G):
    ctx = dmpt.context(0)
    ws = torch.empty(ctx.workspace_size(n, 0, dmpt.options(ckpt_every=1)) + 256, dtype=torch.uint8,
                     device=DEV)
    _, _, info = ctx.sp2_response(levels(n, n // 2), None, n // 2, ckpt_every=1, workspace=ws)
    assert info.converged and info.d0_layer == 1
    return ctx.sp2_backward(G, ws)


@pytest.mark.parametrize("n", [160, 257])
def test_adjoint_start_and_output_are_rounded_once(n):
    G = values(n * n, 126, n + 1).reshape(n, n).to(DEV)
    if n % 2 == 0:                      # symmetric: the ties stay ties
        G = G.triu() + G.triu(1).T
    G[3, 5] = G[5, 3] = (2 - 2.0 ** -24) * 2.0 ** 127 * (1 - 2.0 ** -53)   # rounds down to the largest
    want = (0.5 * (G + G.T)).to(torch.float32).to(F64)
    assert torch.isfinite(want).all()
    assert torch.equal(adjoint(n, G), -want)


@pytest.mark.parametrize("bad", [(2 - 2.0 ** -24) * 2.0 ** 127, 2.0 ** 128, float("inf"),
                                 float("-inf"), float("nan")])
def test_values_that_round_to_infinity_are_refused(bad):
    n = 96
    G = torch.ones(n, n, dtype=F64, device=DEV)
    G[7, 60] = G[60, 7] = bad
    with pytest.raises(dmpt.DmptError) as e:
        adjoint(n, G)
    assert e.value.status == 4
