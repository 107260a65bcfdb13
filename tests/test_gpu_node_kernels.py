"""The per-node FP64 kernels whose obstacle terms are shared by four lanes: the
right-hand side, the auxiliary Dirichlet data, the energy and the boundary
velocity, for obstacle counts around the lane count (0, 1, 4, 5) and node counts
that end inside a CTA.

Tolerances: each quantity is a sum of at most 5 obstacle terms of size <= 1 in
FP64 with a few roundings each (1e-15 of the largest term); 1e-13 of the
largest entry leaves two digits for the library functions and cancellation.
The energy and the boundary velocity follow a double-float pass (2^-48 per
product, ~1e-13 after the spectral derivative), bounded by 1e-10."""
import numpy as np
import pytest

import workloads as W
from oracle import bie as O

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    import paper_2108_01786_gb300 as P
    from paper_2108_01786_gb300 import _build
    _build.build()
    return P


def _geometry(nobs, M0, M1, Me):
    surf = W.fourier_graph(M0, 0.0, np.array([0.08, 0.02]), np.array([0.03, 0.0]))
    bot = W.graph_curve(M1, lambda a: -1.0 + 0 * a, lambda a: 0 * a, lambda a: 0 * a)
    ells = [(0.6 + 1.2 * j, -0.5 - 0.02 * j, 0.15, 0.1, 0.3 * j) for j in range(nobs)]
    g = W.assemble_geometry([surf, bot] + [W.ellipse(Me + j, *e) for j, e in enumerate(ells)], ells)
    f = W.Flow(V1=0.8, a=np.array([0.4, -0.3, 0.2, 0.5, -0.1])[:nobs])
    return g, f, W.filtered_noise(np.random.default_rng(nobs), M0, 0.05, 8)


@pytest.mark.parametrize("nobs,M0,M1,Me", [(0, 65, 49, 40), (1, 97, 61, 45), (4, 130, 64, 51), (5, 127, 66, 48)])
def test_node_kernels_match_oracle(P, nobs, M0, M1, Me):
    import torch
    g, f, ph = _geometry(nobs, M0, M1, Me)
    om_ref, U_ref, _ = O.solve(g, f, ph)
    prob = P.Problem(g, f, ph)
    try:
        prob.assemble("fp64")
        prob.solve()
        b = torch.full((g.N,), np.nan, dtype=torch.float64, device="cuda")
        P.bie_rhs(prob.ctx, prob.phit, b)
        ref = O.rhs(g, f, ph)
        assert np.abs(b.cpu().numpy() - ref).max() <= 1e-13 * np.abs(ref).max()
        Ud = torch.as_tensor(U_ref, device="cuda")
        P.bie_pressure_rhs(prob.ctx, prob.phit, Ud, b, tau=0.07, g=1.0)
        ref = O.pressure_rhs(g, f, ph, U_ref, tau=0.07, g=1.0)
        assert np.abs(b.cpu().numpy() - ref).max() <= 1e-13 * np.abs(ref).max()
        omd = torch.as_tensor(om_ref, device="cuda")
        E = P.bie_energy(prob.ctx, prob.phit, omd, tau=0.07, g=1.0)
        E_ref = O.energy(g, f, ph, om_ref, tau=0.07, g=1.0)
        assert abs(E - E_ref) <= 1e-10 * abs(E_ref)
        fv = torch.empty(g.N, dtype=torch.complex128, device="cuda")
        P.bie_boundary_velocity(prob.ctx, omd, fv)
        ref = np.concatenate(O.boundary_dphi(g, f, om_ref))
        assert np.abs(fv.cpu().numpy() - ref).max() <= 1e-10 * np.abs(ref).max()
        assert np.linalg.norm(prob.U.cpu().numpy() - U_ref) <= 1e-11 * np.linalg.norm(U_ref)
    finally:
        prob.close()
