"""The FP64 transforms (csrc/dft.cu) at the lengths where their forms change: two
steps and direct sums in either pass, one factor above 64, primes on both sides
of Bluestein's threshold (M times its largest prime above 2^20), odd and even.

bie_filter is a forward and an inverse transform with a real symbol <= 1: errors of
a few units of 1e-16 log2(M) of the largest value, 1e-13 bounds them.  The
derivative in bie_pressure_rhs amplifies rounding by |k| <= M/2: 2e-16 M/2 log2(M) of
phi~'s size, below 2e-11 at M = 8200."""
import numpy as np
import pytest

import workloads as W
from oracle import bie as O

pytestmark = pytest.mark.gpu

LENGTHS = [8, 9, 11, 31, 64, 67, 97, 128, 254, 509, 512, 1018, 1021, 1031, 1365, 1502, 2062, 3001, 4016, 4099, 4096,
           8190, 8191]


@pytest.fixture(scope="module")
def P():
    import paper_2108_01786_gb300 as P
    from paper_2108_01786_gb300 import _build
    _build.build()
    return P


@pytest.mark.parametrize("M0", LENGTHS)
def test_filter_and_derivative_of_any_length(P, M0):
    import torch
    g = W.simple_channel(M0, 16)
    f = W.Flow(V1=0.6, a=np.zeros(0))
    rng = np.random.default_rng(M0)
    ph = W.filtered_noise(rng, M0, 1.0, min(8, (M0 - 1) // 2))
    prob = P.Problem(g, f, ph)
    try:
        x = rng.standard_normal(M0)
        xd = torch.as_tensor(x, device="cuda").clone()
        P.bie_filter(prob.ctx, xd)
        assert np.abs(xd.cpu().numpy() - O.filter36(x)).max() <= 1e-13 * np.abs(x).max()
        U = W.filtered_noise(rng, M0, 0.3, min(8, (M0 - 1) // 2))
        b = torch.empty(g.N, dtype=torch.float64, device="cuda")
        P.bie_pressure_rhs(prob.ctx, prob.phit, torch.as_tensor(U, device="cuda"), b, tau=0.1, g=1.0)
        ref = O.pressure_rhs(g, f, ph, U, tau=0.1, g=1.0)
        assert np.abs(b.cpu().numpy() - ref).max() <= 2e-11 * max(1.0, np.abs(ref).max())
    finally:
        prob.close()


def test_several_vectors_of_prime_lengths(P):
    """Batched transforms (one launch for all right-hand sides) with Bluestein blocks."""
    import torch
    g, f, _ = W.random_geometry(np.random.default_rng(3), 4 * 1031)
    assert g.M[0] == 2062 and g.M[1] == 1031
    PH = np.stack([W.filtered_noise(np.random.default_rng(k), g.M[0], 0.05, 8 + k) for k in range(3)])
    prob = P.Problem(g, f, PH[0])
    try:
        prob.assemble("fp16_ir")
        om = torch.empty((3, g.N), dtype=torch.float64, device="cuda")
        U = torch.empty((3, g.M[0]), dtype=torch.float64, device="cuda")
        P.bie_solve_multi(prob.ctx, torch.as_tensor(PH, device="cuda").contiguous(), om, U)
        V = torch.empty(g.M[0], dtype=torch.float64, device="cuda")
        for r in range(3):
            P.bie_normal_velocity(prob.ctx, om[r].contiguous(), V)
            assert float((V - U[r]).norm() / V.norm()) <= 1e-11
            Uref = O.normal_velocity(g, f, om[r].cpu().numpy())
            assert np.linalg.norm(V.cpu().numpy() - Uref) <= 1e-11 * np.linalg.norm(Uref)
    finally:
        prob.close()


@pytest.mark.parametrize("M0,M1", [(1021, 16), (1031, 2053), (2062, 9), (4093, 64)])
def test_context_free_velocity_of_prime_lengths(P, M0, M1):
    """The context-free call sums prime lengths directly, longer ones in pieces of 512 with a
    remainder (1031, 2053, 4093) or not at all (1021)."""
    import torch
    g = W.simple_channel(M0, M1)
    om = W.smooth_density(g, seed=2, kmax=4)
    c = lambda v: torch.as_tensor(np.asarray(v, dtype=complex), device="cuda")
    U = torch.empty(M0, dtype=torch.float64, device="cuda")
    P.bie_normal_velocity_static(list(g.M), c(g.zeta), c(g.dzeta), c(g.d2zeta), None, 0.6, None,
                                 torch.as_tensor(om, device="cuda"), U)
    ref = O.normal_velocity(g, W.Flow(V1=0.6, a=np.zeros(0)), om)
    assert np.linalg.norm(U.cpu().numpy() - ref) <= 1e-11 * np.linalg.norm(ref)
