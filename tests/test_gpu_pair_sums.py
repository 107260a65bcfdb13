"""The matrix-free pair sums (csrc/pair_sums.cuh) and the packed target kernels at
the edges of their tiles: node counts that end inside 32-node tiles, tiles that
span two boundaries, boundaries shorter than a tile, more sources than one chunk;
target counts around the two per thread and the CTA sizes.

Tolerances: double-float sums carry ~48 bits (4e-15 of the largest terms, which are
~M/2 times the result near the diagonal: 1e-12 at these sizes); 1e-10 of the
largest value also covers the spectral derivative.  FP32 far sums: N terms of
relative error 2^-23 against their sum of magnitudes, below 1e-4 of the largest
value for targets clear of the boundaries; the order of the sources is the same
for every target, so a target's value does not depend on the others."""
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


def _geometry(M0, M1, Mo):
    surf = W.fourier_graph(M0, 0.0, np.array([0.08, 0.02]), np.array([0.03, 0.0]))
    bot = W.graph_curve(M1, lambda a: -1.0 + 0 * a, lambda a: 0 * a, lambda a: 0 * a)
    n = max(1, len(Mo))
    ells = [(6.28 * (j + 0.5) / n, -0.5, 0.14, 0.1, 0.4 * j) for j in range(len(Mo))]
    g = W.assemble_geometry([surf, bot] + [W.ellipse(m, *e) for m, e in zip(Mo, ells)], ells)
    return g, W.Flow(V1=0.7, a=np.linspace(-0.4, 0.5, len(Mo)) if Mo else np.zeros(0))


@pytest.mark.parametrize("M0,M1,Mo", [(64, 32, []), (65, 33, [31]), (97, 61, [45, 73]), (256, 128, [64, 64]),
                                       (301, 200, [20, 21, 22, 23])])
def test_boundary_sums_match_oracle(P, M0, M1, Mo):
    import torch
    g, f = _geometry(M0, M1, Mo)
    ph = W.filtered_noise(np.random.default_rng(1), M0, 0.05, 8)
    om = W.smooth_density(g, seed=2, kmax=4)
    prob = P.Problem(g, f, ph)
    try:
        omd = torch.as_tensor(om, device="cuda")
        v = torch.empty(g.N, dtype=torch.complex128, device="cuda")
        P.bie_boundary_velocity(prob.ctx, omd, v)
        ref = np.concatenate(O.boundary_dphi(g, f, om))
        assert np.abs(v.cpu().numpy() - ref).max() <= 1e-10 * np.abs(ref).max()
        E = P.bie_energy(prob.ctx, prob.phit, omd, tau=0.1, g=1.0)
        assert abs(E - O.energy(g, f, ph, om)) <= 1e-10 * max(1.0, abs(E))
        prob.assemble("fp32_ir")
        P.bie_boundary_potential(prob.ctx, omd, v)
        ref = np.concatenate(O.phi_tilde_boundary(g, om))
        assert np.abs(v.cpu().numpy() - ref).max() <= 1e-10 * np.abs(ref).max()
        # Helsing at points near the boundaries and on nodes
        z = np.concatenate([W.near_boundary_targets(g, 45, seed=3), g.zeta[[0, M0, g.N - 1]]])
        uv = torch.empty(len(z), dtype=torch.complex128, device="cuda")
        P.bie_eval_velocity(prob.ctx, omd, torch.as_tensor(z, device="cuda"), uv, mode=P.VEL_HELSING)
        ref = O.helsing_eval(g, O.boundary_dphi(g, f, om), z)
        assert np.abs(uv.cpu().numpy() - ref).max() <= 1e-9 * np.abs(ref).max()
    finally:
        prob.close()


def test_far_targets_do_not_depend_on_their_neighbours(P):
    import torch
    g, f = _geometry(1200, 500, [130, 131])
    om = W.smooth_density(g, seed=2)
    prob = P.Problem(g, f, np.zeros(g.M[0]))
    try:
        omd = torch.as_tensor(om, device="cuda")
        x = np.linspace(0.0, 6.2, 66000)
        z = torch.as_tensor(x + 1j * (-0.2 - 0.05 * np.cos(40 * x)), device="cuda")

        def far(zz, mode):
            uv = torch.full((zz.numel(),), float("nan"), dtype=torch.complex128, device="cuda")
            P.bie_eval_velocity(prob.ctx, omd, zz.contiguous(), uv, mode=mode, near_spacings=1e-6)
            return uv
        full = far(z, P.VEL_FAR)            # 128-thread CTAs
        assert torch.equal(full, far(z, P.VEL_AUTO))
        for n in (1, 2, 31, 32, 33, 63, 64, 65, 129, 1000, 65535):   # one-warp CTAs
            assert torch.equal(far(z[:n], P.VEL_FAR), full[:n]), n
        assert torch.equal(far(z[5:70], P.VEL_FAR), full[5:70])
        ref = O.velocity_far(g, f, om, z[:200].cpu().numpy())
        assert np.abs(full[:200].cpu().numpy() - ref).max() <= 1e-4 * np.abs(ref).max()
    finally:
        prob.close()


@pytest.mark.parametrize("M0,M1,Mo", [(8, 16, []), (9, 8, [15]), (15, 40, [9, 8]), (64, 15, [16, 8]), (16, 17, [8])])
def test_boundary_sums_of_short_boundaries(P, M0, M1, Mo):
    """Boundaries of 8 to 17 nodes, first, last and between: shorter than half a tile."""
    import torch
    g, f = _geometry(M0, M1, Mo)
    om = W.smooth_density(g, seed=2, kmax=2)
    ph = W.filtered_noise(np.random.default_rng(1), M0, 0.05, 2)
    prob = P.Problem(g, f, ph)
    try:
        omd = torch.as_tensor(om, device="cuda")
        v = torch.empty(g.N, dtype=torch.complex128, device="cuda")
        P.bie_boundary_velocity(prob.ctx, omd, v)
        ref = np.concatenate(O.boundary_dphi(g, f, om))
        assert np.abs(v.cpu().numpy() - ref).max() <= 1e-10 * np.abs(ref).max()
        E = P.bie_energy(prob.ctx, prob.phit, omd, tau=0.1, g=1.0)
        assert abs(E - O.energy(g, f, ph, om)) <= 1e-10 * max(1.0, abs(E))
        prob.assemble("fp32_ir")
        P.bie_boundary_potential(prob.ctx, omd, v)
        ref = np.concatenate(O.phi_tilde_boundary(g, om))
        assert np.abs(v.cpu().numpy() - ref).max() <= 1e-10 * np.abs(ref).max()
    finally:
        prob.close()
