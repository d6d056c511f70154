"""Parity of the CUDA adjoint (through the C ABI) with the PyTorch-autograd oracle of the
steady residual operator (oracle/adjoint.py).

Tolerance: FP64, 1e-10 relative to the largest entry of each compared block.  The
steady residual and its VJP are sums of a few hundred terms per entry, evaluated in
a different order on each side; the limiter's min/max choices are taken on values
that agree to ~1e-16, far from a tie on these seeded states.  The adjoint solve is
compared at the tolerance the GMRES is run to.
"""
import dataclasses

import numpy as np
import pytest
import torch

from oracle.adjoint import DRAG, HEAT, Steady
from paper_2303_10846_gb300 import inputs as I
from tests import workloads as TW

pytestmark = pytest.mark.gpu

TOL = 1e-10


def _rel(a, b):
    a, b = np.asarray(a), np.asarray(b)
    return float(np.max(np.abs(a - b)) / max(np.max(np.abs(b)), 1e-300))


def lid_farfield():
    wl = TW.tiny_cavity()
    wl.bcs = [wl.bcs[0], I.BC(I.BC_FARFIELD, 1.05, (0.15, 0.02, -0.03), 1.1)]
    return wl


def tet():
    wl = TW.tiny_tet(n_gh=5, lim=1, cfl_imp=20.0)       # K = 125: ragged tail of 32
    wl.params = dataclasses.replace(wl.params, first_order_iters=0)
    return wl


def tet_sutherland():
    wl = tet()
    wl.params = dataclasses.replace(wl.params, viscosity_law=1, sutherland_c=0.4)
    return wl


WORKLOADS = {"lid_farfield": lid_farfield, "tet": tet, "tet_sutherland": tet_sutherland}


def _solver_prec(wl, prec, m):
    from paper_2303_10846_gb300.rykov import Solver
    s = Solver(wl, prec)
    s.bind_adjoint(m)
    return s


def _solver(wl, m=20):
    return _solver_prec(wl, "fp64", m)


def _blocks(st, x):
    n1 = 2 * st.N * st.K
    return x[:n1], x[n1:n1 + 6 * st.N], x[n1 + 6 * st.N:]


@pytest.mark.parametrize("name", list(WORKLOADS))
def test_steady_residual_vjp_and_objectives(name):
    wl = WORKLOADS[name]()
    s = _solver(wl)
    s.iterate(4)
    x = s.get_state()
    st = Steady(wl)
    xt = torch.as_tensor(x)
    # state round trip through the ABI
    s.put_state(x)
    assert np.array_equal(s.get_state(), x)
    # R(X; p): the blocks are differences of O(1) terms (collision and flux, moments
    # and the state), so the error is measured on the scale of those terms
    r_gpu = s.steady_residual()
    r_orc = st.R_flat(xt, st.p0()).numpy()
    phi, W, q = st.unpack(xt)
    Fm, _ = st.micro_flux(phi, st.p0())
    scales = (float(Fm.abs().max()), float(W.abs().max()), float(W.abs().max()))
    for a, b, sc in zip(_blocks(st, r_gpu), _blocks(st, r_orc), scales):
        assert np.max(np.abs(a - b)) < TOL * sc
    # (dR/dX)^T v and (dR/dp)^T v for a seeded v
    rng = np.random.default_rng(11)
    v = rng.standard_normal(x.size)
    out, pp = s.vjp(v)
    ot, pt = st.vjp(xt, torch.as_tensor(v))
    for a, b in zip(_blocks(st, out), _blocks(st, ot.numpy())):
        assert _rel(a, b) < TOL
    assert _rel(pp, pt.numpy()) < TOL
    # objectives: J, dJ/dX, dJ/dp|_X
    for which, code in (("heat", HEAT), ("drag", DRAG)):
        J, g, dp = s.objective(which)
        Jt, gt, dpt = st.objective_grad(xt, code)
        assert abs(J - Jt) <= 1e-12 * abs(Jt)
        assert _rel(g, gt.numpy()) < TOL
        assert _rel(dp, dpt.numpy()) < TOL


def test_vjp_is_linear_and_padding_free():
    """(dR/dX)^T (a v + b w) = a (dR/dX)^T v + b (dR/dX)^T w, and repeated calls give
    identical bits (fixed-order gathers, no atomics)."""
    wl = tet()
    s = _solver(wl)
    s.iterate(3)
    rng = np.random.default_rng(3)
    v, w = rng.standard_normal(s.state_len), rng.standard_normal(s.state_len)
    ov, _ = s.vjp(v)
    ow, _ = s.vjp(w)
    ovw, _ = s.vjp(2.0 * v - 3.0 * w)
    assert _rel(ovw, 2.0 * ov - 3.0 * ow) < 1e-12
    ov2, _ = s.vjp(v)
    assert np.array_equal(ov, ov2)


def test_adjoint_solve_matches_dense_oracle():
    """Converged steady state on the GPU, GMRES adjoint on the GPU; the oracle solves
    the same transposed system densely at the GPU's state."""
    wl = lid_farfield()
    s = _solver(wl, m=30)
    rc, n, res = s.iterate(3000, 1e-13)
    assert rc == 0 and np.max(res) < 1e-13
    x = s.get_state()
    st = Steady(wl)
    xt = torch.as_tensor(x)
    A = st.jacobian(xt).numpy()
    for which, code in (("heat", HEAT), ("drag", DRAG)):
        it, rel, J, dJdp = s.adjoint_solve(which, max_iter=400, tol=1e-11)
        assert rel <= 1e-11, (which, it, rel)
        Jt, jx, jp = st.objective_grad(xt, code)
        lam_t = np.linalg.solve(A.T, -jx.numpy())
        _, rp = st.vjp(xt, torch.as_tensor(lam_t))
        dJdp_t = (jp + rp).numpy()
        lam = s.adjoint_get()
        assert _rel(lam, lam_t) < 1e-7
        assert _rel(dJdp, dJdp_t) < 1e-8
        assert abs(J - Jt) <= 1e-12 * abs(Jt)
        # warm start: a second call at the same state converges at once
        it2, rel2, _, dJdp2 = s.adjoint_solve(which, max_iter=400, tol=1e-11)
        assert it2 == 0 and rel2 <= 1e-11
        assert _rel(dJdp2, dJdp) < 1e-12


def test_autograd_function_gives_the_adjoint_gradient():
    from paper_2303_10846_gb300.rykov import steady_objective
    wl = lid_farfield()
    s = _solver(wl, m=30)
    st = Steady(wl)
    p = st.p0().clone().requires_grad_(True)
    J = steady_objective(s, p, "heat", n_iter=3000, tol=1e-13, adj_iter=400, adj_tol=1e-11)
    J.backward()
    _, _, J2, dJdp = s.adjoint_solve("heat", max_iter=400, tol=1e-11)
    assert abs(float(J) - J2) <= 1e-12 * abs(J2)
    assert _rel(p.grad.numpy(), dJdp) < 1e-12


def test_adjoint_of_a_mixed_precision_context(monkeypatch):
    """A mixed context's adjoint at its (FP32-distribution) state.  With FP64 arithmetic
    (RYKOV_ADJ_FP64=1) the VJP equals the oracle's at that state to 1e-10; with the
    default FP32 per-velocity arithmetic (compensated velocity sums) to 1e-5; the
    FP32 adjoint solve gives dJ/dp within 1e-4 of the FP64 context's (the two steady
    states differ at the mixed-precision level)."""
    wl = lid_farfield()
    sm = _solver_prec(wl, "mixed", 30)
    rc, n, res = sm.iterate(400, 1e-9)
    assert rc == 0
    x = sm.get_state()
    st = Steady(wl)
    xt = torch.as_tensor(x)
    v = np.random.default_rng(4).standard_normal(x.size)
    ot, pt = st.vjp(xt, torch.as_tensor(v))
    monkeypatch.setenv("RYKOV_ADJ_FP64", "1")
    out, pp = sm.vjp(v)
    for a, b in zip(_blocks(st, out), _blocks(st, ot.numpy())):
        assert _rel(a, b) < TOL
    assert _rel(pp, pt.numpy()) < TOL
    monkeypatch.delenv("RYKOV_ADJ_FP64")
    out32, pp32 = sm.vjp(v)
    for a, b in zip(_blocks(st, out32), _blocks(st, ot.numpy())):
        assert _rel(a, b) < 1e-5
    assert _rel(pp32, pt.numpy()) < 1e-5
    it, rel, J, dJdp = sm.adjoint_solve("heat", max_iter=400, tol=1e-6)
    assert rel <= 1e-6
    s64 = _solver(wl, 30)
    s64.iterate(3000, 1e-13)
    _, _, J64, dJdp64 = s64.adjoint_solve("heat", max_iter=400, tol=1e-10)
    assert abs(J - J64) <= 1e-4 * abs(J64)
    assert _rel(dJdp, dJdp64) < 1e-4


def test_vjp_with_frozen_limiter():
    """After the iteration froze the limiter, the steady operator and its VJP use the
    stored limiter values as constants (the oracle is given the C oracle's values,
    computed from a state equal to the GPU's to round-off)."""
    import oracle as O
    wl = tet()
    wl.params = dataclasses.replace(wl.params, limiter_freeze=5)
    o = O.Oracle(wl)
    o.iterate(8)
    s = _solver(wl)
    s.iterate(8)
    x = s.get_state()
    xt = torch.as_tensor(x)
    st = Steady(wl, L_frozen=o.get(O.BUF_LSTORE))
    r_gpu = s.steady_residual()
    r_orc = st.R_flat(xt, st.p0()).numpy()
    phi, W, q = st.unpack(xt)
    Fm, _ = st.micro_flux(phi, st.p0())
    assert np.max(np.abs(r_gpu[:2 * st.N * st.K] - r_orc[:2 * st.N * st.K])) < 1e-9 * float(Fm.abs().max())
    v = np.random.default_rng(2).standard_normal(x.size)
    out, pp = s.vjp(v)
    ot, pt = st.vjp(xt, torch.as_tensor(v))
    for a, b in zip(_blocks(st, out), _blocks(st, ot.numpy())):
        assert _rel(a, b) < 1e-9


@pytest.fixture(scope="module")
def sphere_first_order():
    """The sphere (61,911 tetrahedra x 3,033 velocities, Mach 5, Kn 0.1) with the
    first-order reconstruction: the limited operator's iteration settles into a limit
    cycle at ~1e-6 (the limiter's min/max selections keep switching), the first-order
    one converges to round-off, so its steady states can be re-converged for finite
    differences."""
    wl = I.sphere_workload()
    wl.params = dataclasses.replace(wl.params, limiter=2)
    return wl


def test_adjoint_sphere_converges_and_matches_finite_differences(sphere_first_order):
    """The adjoint at the sphere's size (the adjoint configuration): rk_adjoint_solve,
    preconditioned by the transposed linearised forward step (micro and macro sweeps),
    reaches a relative residual of 1e-8 for the wall heat and the drag, and dJ/dp with
    respect to (T_w, rho_inf, U_inf,x, T_inf) matches central differences of
    re-converged FP64 steady states (h = 1e-5 of the parameter's scale, residual
    1e-13) within 1e-6 of the largest |dJ/dp|; the mixed context's dJ/dp (its own
    steady state and FP32 adjoint arithmetic) meets the same differences within 1e-6."""
    from paper_2303_10846_gb300.rykov import Solver
    wl = sphere_first_order
    s = Solver(wl, "fp64", params=wl.params)
    rc, n, res = s.iterate(800, tol=1e-13)
    assert rc == 0 and np.max(res) < 1e-13, (n, res)
    s.bind_adjoint(20)
    base = s.get_state()
    adj = {}
    for obj in ("heat", "drag"):
        it, rel, J, dJdp = s.adjoint_solve(obj, max_iter=200, tol=1e-10)
        assert rel <= 1e-8, (obj, it, rel)
        adj[obj] = (J, np.asarray(dJdp))
    ff = [bc for bc in wl.bcs if bc.kind == I.BC_FARFIELD][0]
    p0 = np.array([0.0, ff.rho, ff.U[0], ff.U[1], ff.U[2], ff.T])
    fd = {"heat": np.zeros(6), "drag": np.zeros(6)}
    # re-convergence with a large constant implicit step (the steady state does not
    # depend on it; the first-order iteration stays stable there)
    s.set_params(dataclasses.replace(wl.params, cfl_imp=1000.0, cfl_imp0=0.0, cfl_ramp=1.0))
    for idx in (0, 1, 2, 5):
        h = 1e-5 * max(1.0, abs(p0[idx]))
        vals = []
        for sgn in (1.0, -1.0):
            p = p0.copy()
            p[idx] += sgn * h
            s.put_state(base)
            s.set_boundary_params(p)
            rc, n, res = s.iterate(600, tol=1e-13)
            assert rc == 0 and np.max(res) < 1e-13
            vals.append({o: s.objective(o)[0] for o in ("heat", "drag")})
        for o in ("heat", "drag"):
            fd[o][idx] = (vals[0][o] - vals[1][o]) / (2.0 * h)
    s.put_state(base)
    s.set_boundary_params(p0)
    s.set_params(wl.params)
    for o in ("heat", "drag"):
        g = adj[o][1]
        scale = np.max(np.abs(g))
        for idx in (0, 1, 2, 5):
            assert abs(g[idx] - fd[o][idx]) <= 1e-6 * scale, (o, idx, g[idx], fd[o][idx])
    s.close()
    # the mixed context (FP32 distributions and per-velocity adjoint arithmetic): its
    # steady state stops at a residual of ~6e-8 and its adjoint Krylov solve at ~1e-6
    # (FP32 rounding of the VJP); its dJ/dp still meets the same finite differences
    # within 1e-6 (measured 7e-8 from the FP64 context's dJ/dp)
    m = Solver(wl, "mixed", params=wl.params)
    m.iterate(1500, tol=1e-13)
    m.bind_adjoint(20)
    for o in ("heat", "drag"):
        it, rel, J, dJdp = m.adjoint_solve(o, max_iter=200, tol=1e-10)
        assert rel <= 1e-5, (o, it, rel)
        g, g64 = np.asarray(dJdp), adj[o][1]
        scale = np.max(np.abs(g64))
        assert np.max(np.abs(g - g64)) <= 1e-6 * scale, (o, g, g64)
        for idx in (0, 1, 2, 5):
            assert abs(g[idx] - fd[o][idx]) <= 1e-6 * scale, (o, idx, g[idx], fd[o][idx])
    m.close()


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_adjoint_solve_without_an_iteration_before_it(prec):
    """put_state and a bounded solve on a context that never iterated, its workspace full of
    NaN before the bind, and on two that iterated elsewhere (one of them with a state set
    after that): the same bits."""
    from paper_2303_10846_gb300.rykov import _ptr
    wl = tet()
    donor = _solver_prec(wl, prec, 4)
    donor.iterate(4)
    x = donor.get_state()
    out = []
    for before in ("nothing", "another field", "a field set"):
        s = _solver_prec(wl, prec, 4)
        if before == "nothing":
            s.workspace.fill_(255)
            s._check(s.L.rk_bind_workspace(s.h, _ptr(s.workspace), s.workspace.numel()))
            s.bind_adjoint(4)
        else:
            prim = wl.prim0.copy()
            prim[:, 0] *= 2.0
            prim[:, 4:6] *= 3.0
            s.set_state_prim(prim)
            s.iterate(3)
            if before == "a field set":
                s.set_state_prim(wl.prim0)
        s.put_state(x)
        it, rel, J, dJdp = s.adjoint_solve("heat", max_iter=6, tol=1e-14)
        assert it == 6 and np.isfinite(rel)
        out.append((s.adjoint_get(), np.array([rel, J]), dJdp))
    for a, b, c in zip(*out):
        assert np.array_equal(a, b) and np.array_equal(a, c)


def test_mixed_adjoint_at_grazing_velocities(monkeypatch):
    """Velocities along a wall face whose u.n rounds to a positive number in FP32 and is not
    positive in FP64 (and the other way round): the boundary kernel and the gather have to
    take the same side, or the gather reads what an earlier call left in its scratch."""
    wl = TW.tiny_tet(n_gh=4, lim=2, cfl_imp=20.0)
    m, rng = wl.mesh, np.random.default_rng(2)
    wall = np.nonzero(m.face_cell[:, 1] == -1)[0]
    f32 = np.float32
    extra, kinds = [], set()
    for f in wall:
        n = m.face_normal[f]
        for _ in range(4):
            u = np.cross(n, rng.normal(size=3))
            d64 = (u[0] * n[0] + u[1] * n[1]) + u[2] * n[2]
            a, b = u.astype(f32), n.astype(f32)
            d32 = f32(f32(a[0] * b[0]) + f32(a[1] * b[1])) + f32(a[2] * b[2])
            if (d64 > 0) != (d32 > 0):
                extra.append(u)
                kinds.add(bool(d32 > 0))
    assert len(kinds) == 2
    wl.dvs = I.DVS(u=np.concatenate([wl.dvs.u, extra]),
                   w=np.concatenate([wl.dvs.w, np.full(len(extra), 1e-3 * wl.dvs.w.mean())]))
    s = _solver_prec(wl, "mixed", 2)
    s.iterate(2)
    v = rng.standard_normal(s.state_len)
    out, pp = s.vjp(v)
    s.steady_residual()                           # fills the scratch with FP64 face values
    again, pp2 = s.vjp(v)
    assert np.isfinite(out).all() and np.array_equal(out, again) and np.array_equal(pp, pp2)
    monkeypatch.setenv("RYKOV_ADJ_FP64", "1")
    out64, _ = s.vjp(v)
    st = Steady(wl)
    for a, b in zip(_blocks(st, out), _blocks(st, out64)):
        assert _rel(a, b) < 1e-5


def test_mixed_boundary_terms_are_fp64_and_rounded_once(monkeypatch):
    """First order, so that the face values are the state's in both arithmetics: (dR/dp)^T v
    comes from the boundary kernel alone, FP64 on the FP64 vector (1e-12: the order of the
    operations); dJ/dphi of a cell with one wall face is that face's adjoint, rounded to
    FP32 once (2^-24 of every entry)."""
    wl = TW.tiny_tet(n_gh=5, lim=2, cfl_imp=20.0)
    s = _solver_prec(wl, "mixed", 2)
    s.iterate(3)
    v = np.random.default_rng(6).standard_normal(s.state_len)
    _, pp = s.vjp(v)
    _, g, dp = s.objective("heat")
    monkeypatch.setenv("RYKOV_ADJ_FP64", "1")
    _, pp64 = s.vjp(v)
    _, g64, dp64 = s.objective("heat")
    assert np.abs(pp - pp64).max() <= 1e-12 * np.abs(pp64).max()
    assert np.abs(dp - dp64).max() <= 1e-12 * np.abs(dp64).max()
    fc = wl.mesh.face_cell
    one = np.bincount(fc[fc[:, 1] == -1, 0], minlength=s.N) == 1
    a, b = (x[:2 * s.N * s.K].reshape(2, s.N, s.K)[:, one] for x in (g, g64))
    assert one.sum() > 10 and np.abs(b).max() > 0
    assert (np.abs(a - b) <= 2.0 ** -24 * (1 + 1e-6) * np.abs(b)).all()


@pytest.mark.parametrize("prec,b", [("mixed", 18), ("mixed", -12), ("fp64", 18)])
def test_adjoint_product_in_other_units_of_velocity(prec, b):
    """Velocities times c = 2^b (the gas constant, the viscosity and the weights with them;
    18: metres to some hundredths of a millimetre per second): the products of the two unit
    systems agree to the tolerances of the precisions.  X scales as (c^-3 | 1, c, c, c, c^2,
    c^2 | c^3), R as (c^-2 | as X | as X), the product of v/R as 1/X; first order (the FP32
    limiter derivative has an absolute threshold)."""
    import copy
    base = TW.tiny_tet(n_gh=5, lim=2, cfl_imp=20.0)
    wl = copy.deepcopy(base)
    c = 2.0 ** b
    wl.prim0[:, 1:4] *= c
    wl.dvs = I.DVS(u=base.dvs.u * c, w=base.dvs.w * c ** 3)
    wl.params.R *= c * c
    wl.params.mu_ref *= c
    wl.bcs = [I.BC(q.kind, q.rho, tuple(x * c for x in q.U), q.T) for q in base.bcs]
    s = _solver_prec(base, prec, 2)
    s.iterate(3)
    N, K = s.N, s.K
    tail = np.concatenate([np.tile([1.0, c, c, c, c * c, c * c], N), np.full(6 * N, c ** 3)])
    X = np.concatenate([np.full(2 * N * K, c ** -3), tail])
    X[N * K:2 * N * K] = c ** -1
    R = np.concatenate([np.full(2 * N * K, c ** -2), tail])
    R[N * K:2 * N * K] = 1.0
    v = np.random.default_rng(12).standard_normal(s.state_len)
    out, _ = s.vjp(v)
    t = _solver_prec(wl, prec, 2)
    t.put_state(s.get_state() * X)
    scaled, _ = t.vjp(v / R)
    st = Steady(base)
    for p, q in zip(_blocks(st, scaled * X), _blocks(st, out)):
        assert _rel(p, q) < (1e-10 if prec == "fp64" else 1e-5)


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("name", ["tet", "lid_farfield"])
def test_adjoint_workspace_size(name, prec):
    """In vectors of 2 N K_pad doubles: two face arrays, the neighbours' shares (one a face of
    a cell) with the preconditioner's two temporaries inside them, five vectors, the staging,
    the inverse diagonal (1/2), the Krylov space, and of mixed contexts two copies of the
    state and an FP32 vector; and some 200 doubles a cell of records (faces shared by two)."""
    import ctypes as C
    wl = WORKLOADS[name]()
    s = _solver_prec(wl, prec, 4)
    m = wl.mesh
    ms = np.bincount(m.face_cell[m.face_cell >= 0].ravel()).max()
    for k in (1, 20):
        n = C.c_size_t()
        s._check(s.L.rk_adjoint_workspace_size(s.h, k, C.byref(n)))
        fields = 2 * m.n_face / m.n_cell + ms + 5 + 1 + 0.5 + (k + 1) + (2.5 if prec == "mixed" else 0)
        records = 60 * ms + 300
        fixed = 8 * (1024 * 64 + 4096) + 40 * 256
        assert n.value <= 8 * s.N * (2 * s.Kp * fields + records + 12 * (k + 7)) + fixed
