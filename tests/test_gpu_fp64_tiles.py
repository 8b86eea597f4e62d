"""FP64 layer kernel at the edges of its tiles: sizes on both sides of a tile
edge, of a K block (16) and of the sizes where the tile grows (8 up to n = 400,
16 up to 2048, 32 above), against the FP64 oracle.

Tolerance: 1e-10 relative, that of the FP64 form (its sums of at most 2n
products of values within [-1.25, 1.25] round to a few n 2^-53, amplified by
(eps_N - eps_1) / gap < 1e3 here).
"""

import numpy as np
import pytest
import torch

import oracle
from paper_2203_09621_gb300 import dmpt
from paper_2203_09621_gb300.workloads import make_instance

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    return dmpt.context(0)


@pytest.mark.parametrize("n,k,ld", [(2, 1, 2), (7, 2, 7), (8, 1, 11), (9, 1, 9), (17, 3, 17),
                                    (400, 1, 400), (401, 2, 408), (641, 1, 641), (2049, 1, 2049)])
def test_fp64_tile_edges(ctx, n, k, ld):
    inst = make_instance(f"fp64-n{n}", n, (n + 1) // 2, (-2.0, -0.25), (0.25, 2.0), "gauss", k,
                         0.01, seed=640 + n)
    H = torch.zeros(n, ld, dtype=torch.float64, device="cuda")[:, :n]
    H1 = torch.zeros(k, n, ld, dtype=torch.float64, device="cuda")[:, :, :n]
    H.copy_(torch.from_numpy(inst.H))
    H1.copy_(torch.from_numpy(inst.H1))
    P, P1, info = ctx.sp2_response(H, H1, inst.n_occ, precision="fp64")
    assert info.converged
    for j in range(k):
        P_ref, P1_ref = oracle.response_from_eigs(inst.eps, inst.Q, inst.H1[j], inst.n_occ)
        assert np.linalg.norm(P1[j].cpu().numpy() - P1_ref) <= 1e-10 * np.linalg.norm(P1_ref)
    assert np.linalg.norm(P.cpu().numpy() - P_ref) <= 1e-10 * np.linalg.norm(P_ref)
    assert torch.equal(P, P.T) and torch.equal(P1, P1.transpose(1, 2))
