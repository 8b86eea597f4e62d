"""Tile widths of the grouped batch kernels (group_tile_n).

Each width that is asked for runs, the default takes 128 for small instances
and 256 once a large one is in the batch, and every instance whose 256 x 256
tiles take one round of the CTA pairs equals its single solve bit for bit at
both widths.
"""

import pytest

from paper_2203_09621_gb300.workloads import make_instance

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2203_09621_gb300 import dmpt  # noqa: E402

DEV = torch.device("cuda:0")


def batch(sizes, k):
    xs = [make_instance(f"bw{i}", n, max(1, n // 2), (-2.0, -0.1), (0.1, 2.0), seed=9600 + n, k=k)
          for i, n in enumerate(sizes)]
    return ([torch.from_numpy(x.H).to(DEV) for x in xs], [torch.from_numpy(x.H1).to(DEV) for x in xs],
            [x.n_occ for x in xs])


@pytest.mark.parametrize("precision", ["dual_fp16", "dual_bf16"])
@pytest.mark.parametrize("sizes,k,opts", [
    ([2, 31, 33, 64, 129, 255, 257], 1, {}),          # edges of the 32-, 128- and 256-wide blocks
    ([300, 385, 513, 700, 1000], 2, {}),
    ([289, 769, 1025], 3, dict(accum_chunk=96)),
    ([512, 640], 5, dict(tile_band=0)),
])
def test_both_widths_equal_single_solves(precision, sizes, k, opts):
    ctx = dmpt.context(0)
    Hs, H1s, occ = batch(sizes, k)
    single = [ctx.sp2_response(H, H1, o, precision=precision, **opts)
              for H, H1, o in zip(Hs, H1s, occ)]
    for width in (256, 128, 0):
        Ps, P1s, infos = ctx.sp2_response_batch(Hs, H1s, occ, precision=precision,
                                                group_tile_n=width, **opts)
        for n, P, P1, info, (Pr, P1r, ref) in zip(sizes, Ps, P1s, infos, single):
            assert info.layers == ref.layers, (width, n)
            assert torch.equal(P, Pr) and torch.equal(P1, P1r), (width, n)


def test_the_width_that_is_asked_for_runs():
    ctx = dmpt.context(0)
    Hs, H1s, occ = batch([777, 1000], 2)

    def norms(width, Hs=Hs, H1s=H1s, occ=occ):
        infos = ctx.sp2_response_batch(Hs, H1s, occ, group_tile_n=width)[2]
        return [i.n_x + i.froerr1_hist[0] + i.froerr1_hist[1] for i in infos[:2]]

    wide, narrow = norms(256), norms(128)
    # the norms are sums over the tiles: the two widths round them differently
    assert wide != narrow
    assert norms(0) == narrow
    big = batch([1600], 2)                            # more than five blocks of 256
    assert norms(0, Hs + big[0], H1s + big[1], occ + big[2]) == wide


def test_other_widths_are_refused():
    ctx = dmpt.context(0)
    Hs, H1s, occ = batch([64], 1)
    for width in (-1, 1, 64, 512):
        with pytest.raises(dmpt.DmptError) as e:
            ctx.sp2_response_batch(Hs, H1s, occ, group_tile_n=width)
        assert e.value.status == 1
