"""FP32 layer kernel at the edges of its tiles (64 wide while few 128-wide tiles
would run, 128 above): sizes on both sides of a tile edge, of a K block (16) and
of the line between the widths, against the FP64 oracle.

Tolerance: that of the FP32 form in the parity tests,
10 u (eps_N - eps_1) / gap with u = 2^-24.
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


@pytest.mark.parametrize("n,k,ld", [(2, 1, 2), (15, 2, 15), (17, 1, 24), (64, 1, 64), (65, 3, 65),
                                    (129, 1, 129), (896, 2, 896), (897, 2, 897), (1153, 1, 1153)])
def test_fp32_tile_edges(ctx, n, k, ld):
    inst = make_instance(f"fp32-n{n}", n, (n + 1) // 2, (-2.0, -0.25), (0.25, 2.0), "gauss", k,
                         0.01, seed=320 + n)
    H = torch.zeros(n, ld, dtype=torch.float64, device="cuda")[:, :n]
    H1 = torch.zeros(k, n, ld, dtype=torch.float64, device="cuda")[:, :, :n]
    H.copy_(torch.from_numpy(inst.H))
    H1.copy_(torch.from_numpy(inst.H1))
    P, P1, info = ctx.sp2_response(H, H1, inst.n_occ, precision="fp32")
    assert info.converged
    gap = inst.eps[inst.n_occ] - inst.eps[inst.n_occ - 1]
    tol = 10.0 * 2.0 ** -24 * (info.eps_max - info.eps_min) / gap
    for j in range(k):
        P_ref, P1_ref = oracle.response_from_eigs(inst.eps, inst.Q, inst.H1[j], inst.n_occ)
        assert np.linalg.norm(P1[j].cpu().numpy() - P1_ref) <= tol * np.linalg.norm(P1_ref)
    assert np.linalg.norm(P.cpu().numpy() - P_ref) <= tol * np.linalg.norm(P_ref)
    assert torch.equal(P, P.T) and torch.equal(P1, P1.transpose(1, 2))
