"""Tile widths of the pair kernel (256, 128 or 64 columns by size).

A narrow tile is part of a 256 x 256 tile: it keeps that tile's K direction and
accumulation chunks, so a single solve (any width) and the grouped batch kernel
(always 256 wide) give the same bits.  Sizes: the edges of the 64-wide range,
K ranges of odd and partial 32-column blocks, one and several rounds of tiles
(backwards K sweeps), accumulation chunks that do not divide the K range.
"""

import pytest

from paper_2203_09621_gb300.workloads import make_instance

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2203_09621_gb300 import dmpt  # noqa: E402

DEV = torch.device("cuda:0")


def instance(n, k):
    x = make_instance(f"w{n}", n, max(1, n // 2), (-2.0, -0.1), (0.1, 2.0), seed=9700 + n, k=k)
    return torch.from_numpy(x.H).to(DEV), torch.from_numpy(x.H1).to(DEV), x.n_occ


@pytest.mark.parametrize("n,k,opts", [
    (2, 1, {}), (31, 2, {}), (33, 1, {}), (255, 1, {}), (257, 1, {}), (289, 2, {}),
    (512, 5, {}), (513, 5, {}),            # 18 items (64 wide), 36 items (128 wide)
    (769, 3, dict(accum_chunk=96)), (1000, 2, dict(accum_chunk=32)),
    (1281, 3, {}),                         # 84 items: two rounds, 128 wide
    (2081, 2, {}), (2081, 2, dict(accum_chunk=160)), (2081, 2, dict(k_snake=0)),
    (1280, 3, dict(tile_band=0)), (2300, 1, dict(tile_band=3)),
])
def test_single_solve_equals_grouped_kernel(n, k, opts):
    ctx = dmpt.context(0)
    H, H1, n_occ = instance(n, k)
    Ps, P1s, infos = ctx.sp2_response_batch([H, H], [H1, H1], [n_occ, n_occ], **opts)
    P, P1, info = ctx.sp2_response(H, H1, n_occ, **opts)
    torch.cuda.synchronize()
    assert info.converged and infos[0].layers == info.layers
    assert torch.equal(Ps[0], P) and torch.equal(P1s[0], P1)
    assert torch.equal(P, P.T) and torch.equal(P1, P1.transpose(1, 2))


@pytest.mark.parametrize("n,order,k", [(200, 4, 2), (513, 3, 2)])
def test_higher_orders_equal_the_single_cta_kernel(n, order, k):
    ctx = dmpt.context(0)
    H, H1, n_occ = instance(n, k)
    P, terms, _ = ctx.sp2_response_m(H, H1, n_occ, order)
    Pc, termsc, _ = ctx.sp2_response_m(H, H1, n_occ, order, cta_pair=0)
    torch.cuda.synchronize()
    assert torch.equal(P, Pc)
    for a, b in zip(terms, termsc):
        assert torch.equal(a, b)


@pytest.mark.parametrize("n,k,opts", [
    (65, 2, {}), (257, 1, {}), (1000, 2, {}), (1281, 3, {}), (2081, 2, {}),
    (300, 1, dict(cta_pair=0)), (1281, 1, dict(cta_pair=0)), (700, 1, dict(precision="dual_bf16")),
])
def test_padding_of_the_workspace_may_hold_anything(n, k, opts):
    """Elements past the last K block are neither computed nor read as data."""
    ctx = dmpt.context(0)
    H, H1, n_occ = instance(n, k)
    prec = dict(precision=opts["precision"]) if "precision" in opts else {}
    nbytes = ctx.workspace_size(n, k, dmpt.options(**opts))
    P, P1, info = ctx.sp2_response(H, H1, n_occ, **opts)
    for fill in (0xFF, 0x7C):   # NaN in every type; large values
        ws = torch.full((nbytes + 256,), fill, dtype=torch.uint8, device=DEV)
        Pw, P1w, infow = ctx.sp2_response(H, H1, n_occ, workspace=ws, **opts)
        assert infow.converged and infow.layers == info.layers
        assert torch.equal(P, Pw) and torch.equal(P1, P1w)
    Pb, P1b, _ = ctx.sp2_response_batch([H, H], [H1, H1], [n_occ, n_occ], **prec)
    assert torch.equal(Pb[1], P) and torch.equal(P1b[1], P1)
