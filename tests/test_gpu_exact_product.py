"""The exact-slice product (bie_matmat_full) at the edges of its tiles: row blocks
and K tiles with remainders, fewer units than SMs, column counts around the
padding to 16 and around the split into two groups, several pieces per row block.

Tolerance: the storage carries ~2^-48 and the slices are cut below 2^-50 of each
row's and each column's scale, which leaves 1e-13 of sum_l |A_ml| |x_l| / M_l.
"""
import numpy as np
import pytest

import workloads as W
from oracle import bie as O

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    import paper_2108_01786_gb300 as P
    return P


@pytest.mark.parametrize("n,nrhs", [(192, 1), (257, 3), (257, 49), (640, 16), (1001, 17), (1001, 33),
                                    (1600, 48), (1600, 64), (2944, 50)])
def test_matmat_full_edges(P, n, nrhs):
    import torch
    g, f, ph = W.random_geometry(np.random.default_rng(n), n)
    A = O.assemble(g)
    rng = np.random.default_rng(nrhs)
    X = rng.standard_normal((nrhs, g.N)) * 10.0 ** rng.uniform(-9, 9, (nrhs, 1))
    if nrhs > 2:
        X[1] = 0.0                       # an empty column
        X[2, ::2] *= 1e-14               # values below the column's last slices
    prob = P.Problem(g, f, ph)
    try:
        prob.assemble("fp32_ir")
        Xd = torch.as_tensor(X, device="cuda").contiguous()
        Yd = torch.empty_like(Xd)
        P.bie_matmat_full(prob.ctx, Xd, Yd)
        Y = Yd.cpu().numpy()
        scale = np.abs(X) @ np.abs(A).T
        assert np.all(np.abs(Y - X @ A.T) <= 1e-13 * scale)
    finally:
        prob.close()


def test_matmat_full_not_finite(P):
    """A value that is not finite makes its own column NaN and no other."""
    import torch
    g, f, ph = W.random_geometry(np.random.default_rng(3), 640)
    X = np.random.default_rng(4).standard_normal((6, g.N))
    prob = P.Problem(g, f, ph)
    try:
        prob.assemble("fp16_ir")
        want = torch.empty((6, g.N), dtype=torch.float64, device="cuda")
        P.bie_matmat_full(prob.ctx, torch.as_tensor(X, device="cuda"), want)
        X[1, 5], X[4, g.N - 1] = np.nan, np.inf
        got = torch.empty_like(want)
        P.bie_matmat_full(prob.ctx, torch.as_tensor(X, device="cuda"), got)
        assert torch.isnan(got[1]).all() and torch.isnan(got[4]).all()
        for r in (0, 2, 3, 5):
            assert torch.equal(got[r], want[r])
    finally:
        prob.close()
