"""The one-kernel solver (csrc/resident.cu) against the kernel-by-kernel one,
which profiling selects, at the sizes where its row split can go wrong: one CTA,
one row more or less than the row warps take, row counts per CTA off the quads,
all SMs; restart lengths from 1, no obstacles and many, both row signs, initial
guesses, zero and non-finite data.

Both stop at ||r|| <= 1e-14 ||b|| (the caller's rtol where it is larger), so their
solutions differ by at most 2 rtol ||b|| / sigma_min(A) plus rounding; sigma_min >=
0.1 ||A|| on these geometries (spectrum clustered at 1/2): 1e-12 of ||omega|| bounds
it for rtol 1e-14, 100 rtol in general."""
import numpy as np
import pytest

import workloads as W

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
    ells = [(6.28 * (j + 0.5) / n, -0.5 - 0.01 * j, 0.12, 0.1, 0.4 * j) for j in range(len(Mo))]
    g = W.assemble_geometry([surf, bot] + [W.ellipse(m, *e) for m, e in zip(Mo, ells)], ells)
    a = np.linspace(-0.4, 0.5, len(Mo)) if Mo else np.zeros(0)
    return g, W.Flow(V1=0.7, a=a), W.filtered_noise(np.random.default_rng(M0), M0, 0.05, min(8, M0 // 4))


SIZES = [(16, 12, []),                      # one CTA, fewer rows than a quad round
         (20, 11, []),                      # 31 rows: one CTA, every row warp
         (20, 12, []),                      # 32: two CTAs
         (41, 29, [23, 25]),                # 118 rows on 4 CTAs, the last one short
         (150, 81, [40] * 6),               # six obstacles
         (640, 330, [161, 170]),            # 1301 rows
         (2356, 1178, [589, 589]),          # 31 x 152: one row per row warp on every SM
         (2357, 1179, [589, 589])]          # and two more rows


@pytest.mark.parametrize("M0,M1,Mo", SIZES)
@pytest.mark.parametrize("prec", ["fp64", "fp32_ir", "fp16_ir", "bf16_ir"])
def test_one_kernel_solve_equals_the_stepwise_one(P, M0, M1, Mo, prec):
    import torch
    g, f, ph = _geometry(M0, M1, Mo)
    prob = P.Problem(g, f, ph)
    try:
        prob.assemble(prec)
        rng = np.random.default_rng(3)
        b = torch.as_tensor(np.concatenate([W.filtered_noise(rng, m, 0.5, max(1, m // 8)) for m in g.M]), device="cuda")
        for kw in ({}, {"row_flip": 0}, {"restart": 3, "max_cycles": 60, "rtol": 1e-12}, {"restart": 1, "rtol": 1e-4},
                   {"restart": 200}, {"rtol": 1e-10, "inner_tol": 1e-2}):
            o = P.bie_default_opts(**kw)
            res = []
            for prof in (0, 1):
                P.bie_set_profiling(prob.ctx, prof)
                om = torch.full((g.N,), np.nan, dtype=torch.float64, device="cuda")
                try:
                    info, st = P.bie_solve_b(prob.ctx, b, om, o), 0
                except P.BieError as e:
                    info, st = None, e.status
                res.append((st, om.cpu().numpy(), info))
            (s0, x0, i0), (s1, x1, i1) = res
            assert s0 == s1, (kw, s0, s1)
            if s0 == 0:
                assert i0.converged and i0.rel_resid <= o.rtol
                bound = max(1e-12, 100.0 * o.rtol)
                assert np.linalg.norm(x0 - x1) <= bound * np.linalg.norm(x1), kw
    finally:
        prob.close()


@pytest.mark.parametrize("prec", ["fp64", "fp32_ir", "fp16_ir"])
def test_one_kernel_solve_guesses_zero_and_nonfinite(P, prec):
    import torch
    g, f, ph = _geometry(120, 61, [40, 41])
    prob = P.Problem(g, f, ph)
    try:
        prob.assemble(prec)
        prob.solve()
        om = prob.omega.clone()
        # from the solution: nothing to do; from a perturbed one: the same solution
        assert P.bie_solve(prob.ctx, prob.phit, prob.omega, prob.U, None, P.bie_default_opts(x0=1)).cycles <= 1
        prob.omega.copy_(om * (1.0 + 1e-3) + 1e-4)
        info = P.bie_solve(prob.ctx, prob.phit, prob.omega, prob.U, None, P.bie_default_opts(x0=1))
        assert info.converged
        assert float((prob.omega - om).norm() / om.norm()) <= 1e-12
        z = torch.zeros(g.N, dtype=torch.float64, device="cuda")
        for x0 in (0, 1):
            x = torch.ones(g.N, dtype=torch.float64, device="cuda")
            info = P.bie_solve_b(prob.ctx, z, x, P.bie_default_opts(x0=x0))
            assert info.converged and info.iters == 0 and float(x.abs().max()) == 0.0
        z[7] = float("nan")
        with pytest.raises(P.BieError) as e:
            P.bie_solve_b(prob.ctx, z, x)
        assert e.value.status == P.BIE_ERR_NAN
        with pytest.raises(P.BieError) as e:
            P.bie_solve(prob.ctx, prob.phit, prob.omega, prob.U, None, P.bie_default_opts(max_cycles=1, restart=2))
        assert e.value.status == P.BIE_ERR_NOCONV
        assert prob.solve().converged   # the context stays usable
        # tiny and huge data (the solve is linear)
        for s in (1e-30, 1e30):
            info = P.bie_solve(prob.ctx, prob.phit, prob.omega, prob.U, None)
            b = torch.empty(g.N, dtype=torch.float64, device="cuda")
            P.bie_rhs(prob.ctx, prob.phit, b)
            x = torch.empty_like(b)
            info = P.bie_solve_b(prob.ctx, b * s, x)
            assert info.converged
            assert float((x / s - prob.omega).norm() / prob.omega.norm()) <= 1e-12
    finally:
        prob.close()


def test_precision_change_on_one_context(P):
    """The schemes share the solver's exchange buffers, whose padding past N must read as
    zero.  The FP64 solve here leaves doubles whose low words are NaN as floats where
    the refined schemes have their padding: x is the solution already, so x / M_l is
    published once (1 / M_l a power of two keeps the low words) and nothing after it."""
    import torch
    g, f, ph = _geometry(64, 32, [9])
    assert g.N == 105                        # floats 105 .. 127 overlay doubles 52 .. 63, surface nodes
    x = np.random.default_rng(5).standard_normal(g.N)
    low = x.view(np.uint64) & np.uint64(0xffffffff00000000)
    x = (low | np.uint64(0x7fc00001)).view(np.float64)
    xd = torch.as_tensor(x, device="cuda")
    prob = P.Problem(g, f, ph)
    try:
        for prec in ("fp32_ir", "fp16_ir", "bf16_ir"):
            prob.assemble("fp64")
            b = torch.empty_like(xd)
            P.bie_matvec(prob.ctx, 1, xd, b)
            om = xd.clone()
            info = P.bie_solve_b(prob.ctx, b, om, P.bie_default_opts(x0=1, rtol=1e-10))
            assert info.cycles == 0 and torch.equal(om, xd)
            prob.assemble(prec)
            info = P.bie_solve_b(prob.ctx, b, om)
            assert info.converged
            other = P.Problem(g, f, ph)      # a context that never solved in FP64
            try:
                other.assemble(prec)
                want = torch.empty_like(om)
                P.bie_solve_b(other.ctx, b, want)
                assert torch.equal(om, want), prec
            finally:
                other.close()
    finally:
        prob.close()


@pytest.mark.parametrize("n", [1001, 4099])
def test_fp64_then_refined_on_one_context(P, n):
    g, f, ph = W.random_geometry(np.random.default_rng(n), n)
    prob = P.Problem(g, f, ph)
    try:
        for seed in range(6):
            prob.phit.copy_(prob.phit.new_tensor(W.filtered_noise(np.random.default_rng(seed), g.M[0], 0.05, 8)))
            prob.assemble("fp64")
            assert prob.solve().converged
            ref = prob.omega.clone()
            for prec in ("fp32_ir", "fp16_ir", "bf16_ir"):
                prob.assemble(prec)
                assert prob.solve().converged
                assert float((prob.omega - ref).norm() / ref.norm()) <= 1e-12
    finally:
        prob.close()


@pytest.mark.parametrize("prec", ["fp64", "fp32_ir", "fp16_ir", "bf16_ir"])
def test_failed_solve_leaves_U_and_psi_alone(P, prec):
    """A non-finite right-hand side: no iterate, so U and psi keep the caller's values; a solve
    that only missed rtol gives them from its last iterate."""
    import torch
    g, f, ph = _geometry(120, 61, [40, 41])
    prob = P.Problem(g, f, ph)
    try:
        prob.assemble(prec)
        om = torch.empty(g.N, dtype=torch.float64, device="cuda")
        U = torch.full((g.M[0],), 7.0, dtype=torch.float64, device="cuda")
        psi = torch.full((2,), -3.0, dtype=torch.float64, device="cuda")
        bad = prob.phit.clone()
        bad[3] = float("nan")
        for prof in (0, 1):                     # the one-kernel solver, the kernel-by-kernel one
            P.bie_set_profiling(prob.ctx, prof)
            with pytest.raises(P.BieError) as e:
                P.bie_solve(prob.ctx, bad, om, U, psi)
            assert e.value.status == P.BIE_ERR_NAN
            assert bool((U == 7.0).all()) and bool((psi == -3.0).all()), prof
        P.bie_set_profiling(prob.ctx, 0)
        with pytest.raises(P.BieError) as e:
            P.bie_solve(prob.ctx, prob.phit, om, U, psi, P.bie_default_opts(max_cycles=1, restart=2))
        assert e.value.status == P.BIE_ERR_NOCONV
        want = torch.empty_like(U)
        P.bie_normal_velocity(prob.ctx, om, want)
        assert torch.equal(U, want) and bool((psi != -3.0).all())
        assert P.bie_solve(prob.ctx, prob.phit, om, U, psi).converged
    finally:
        prob.close()


def _both_solvers(P, prob, b, N, **kw):
    """(status, x, info) of the one-kernel solver and of the kernel-by-kernel one."""
    import torch
    out = []
    for prof in (0, 1):
        P.bie_set_profiling(prob.ctx, prof)
        om = torch.full((N,), np.nan, dtype=torch.float64, device="cuda")
        try:
            info, st = P.bie_solve_b(prob.ctx, b, om, P.bie_default_opts(**kw)), 0
        except P.BieError as e:
            info, st = None, e.status
        out.append((st, om, info))
    P.bie_set_profiling(prob.ctx, 0)
    return out


@pytest.mark.parametrize("n,prec", [(6655, "fp16_ir"), (6703, "fp16_ir"), (6703, "bf16_ir"), (4740, "fp32_ir"),
                                    (4801, "fp32_ir")])
def test_one_kernel_solve_around_the_l2_size(P, n, prec):
    """Just below and just above 90 MB of inner storage, where a row takes one warp and
    the heads of the rows leave shared memory; ragged sizes."""
    import torch
    g, f, ph = W.random_geometry(np.random.default_rng(n), n)
    assert g.N % 64 != 0
    prob = P.Problem(g, f, ph)
    try:
        prob.assemble(prec)
        b = torch.empty(g.N, dtype=torch.float64, device="cuda")
        P.bie_rhs(prob.ctx, prob.phit, b)
        (s0, x0, i0), (s1, x1, i1) = _both_solvers(P, prob, b, g.N)
        assert s0 == s1 == 0 and i0.converged and i1.converged
        assert float((x0 - x1).norm() / x1.norm()) <= 1e-12
    finally:
        prob.close()


@pytest.mark.parametrize("M0,M1,Mo", [(20, 12, []), (41, 29, [23, 25]), (640, 330, [161, 170])])
@pytest.mark.parametrize("prec", ["fp64", "fp32_ir", "bf16_ir"])
def test_option_sets_that_must_converge_and_that_must_not(P, M0, M1, Mo, prec):
    """The option sets of the comparison that have to converge do, and where both solvers run
    out of cycles their iterates are equally good: residuals within a factor of 2."""
    import torch
    g, f, ph = _geometry(M0, M1, Mo)
    prob = P.Problem(g, f, ph)
    try:
        prob.assemble(prec)
        b = torch.empty(g.N, dtype=torch.float64, device="cuda")
        P.bie_rhs(prob.ctx, prob.phit, b)
        for kw in ({}, {"row_flip": 0}, {"restart": 200}, {"rtol": 1e-10, "inner_tol": 1e-2}):
            for st, _, info in _both_solvers(P, prob, b, g.N, **kw):
                assert st == 0 and info.converged, kw
        y = torch.empty_like(b)
        for kw in ({"restart": 3, "max_cycles": 2}, {"restart": 2, "max_cycles": 3}, {"restart": 5, "max_cycles": 1}):
            res = []
            for st, x, _ in _both_solvers(P, prob, b, g.N, **kw):
                assert st == P.BIE_ERR_NOCONV, kw
                P.bie_matvec(prob.ctx, 1, x, y)
                res.append(float((b - y).norm() / b.norm()))
            assert 1e-13 < max(res) < 1.0 and max(res) <= 2.0 * min(res), (kw, res)
    finally:
        prob.close()


def _many(nobs, M0, M1, Mo):
    surf = W.fourier_graph(M0, 0.0, np.array([0.08, 0.02]), np.array([0.03, 0.0]))
    bot = W.graph_curve(M1, lambda a: -1.0 + 0 * a, lambda a: 0 * a, lambda a: 0 * a)
    r = 1.2 / nobs
    ells = [(6.28 * (j + 0.5) / nobs, -0.5, r, 0.8 * r, 0.4 * j) for j in range(nobs)]
    g = W.assemble_geometry([surf, bot] + [W.ellipse(m, *e) for m, e in zip(Mo, ells)], ells)
    return g, W.Flow(V1=0.7, a=np.linspace(-0.4, 0.5, nobs)), W.filtered_noise(np.random.default_rng(M0), M0, 0.05, 8)


@pytest.mark.parametrize("nobs", [19, 20, 25, 30])
@pytest.mark.parametrize("prec", ["fp32_ir", "bf16_ir"])
def test_many_obstacles_in_the_kernel_by_kernel_solver(P, nobs, prec):
    """As many obstacles as boundaries are allowed: the product has 20 to 32 warps, fewer
    than the obstacles where its chunk of rows needs no more."""
    import torch
    g, f, ph = _many(nobs, 100, 60, [16 + j % 5 for j in range(nobs)])
    prob = P.Problem(g, f, ph)
    try:
        prob.assemble(prec)
        b = torch.empty(g.N, dtype=torch.float64, device="cuda")
        P.bie_rhs(prob.ctx, prob.phit, b)
        for kw in ({}, {"row_flip": 0}):
            (s0, x0, i0), (s1, x1, i1) = _both_solvers(P, prob, b, g.N, **kw)
            assert (s0, s1) == (0, 0) and i0.converged and i1.converged, kw
            assert abs(i0.iters - i1.iters) <= 3
            assert float((x0 - x1).norm() / x1.norm()) <= 1e-12
    finally:
        prob.close()


@pytest.mark.parametrize("nobs,M0,M1,Mo", [(25, 2400, 1200, 48), (30, 2500, 1300, 46), (30, 60, 40, 20), (21, 2400, 1200, 57)])
@pytest.mark.parametrize("prec", ["fp64", "fp32_ir", "fp16_ir"])
def test_more_obstacles_than_row_warps(P, nobs, M0, M1, Mo, prec):
    """4700 to 5200 unknowns: 32 to 35 rows on 20 to 31 row warps per CTA, fewer than the
    obstacles whose sums they reduce (21, 25, 30); a small case with more warps than those."""
    import torch
    g, f, ph = _many(nobs, M0, M1, [Mo + j % 3 for j in range(nobs)])
    prob = P.Problem(g, f, ph)
    try:
        prob.assemble(prec)
        b = torch.empty(g.N, dtype=torch.float64, device="cuda")
        P.bie_rhs(prob.ctx, prob.phit, b)
        for kw in ({}, {"row_flip": 0}):
            (s0, x0, i0), (s1, x1, i1) = _both_solvers(P, prob, b, g.N, **kw)
            assert (s0, s1) == (0, 0) and i0.converged and i1.converged, kw
            assert float((x0 - x1).norm() / x1.norm()) <= 1e-12
    finally:
        prob.close()
