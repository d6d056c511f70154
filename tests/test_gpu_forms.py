"""Kernel forms that the other meshes do not reach: cells with eight faces (the widest
instantiations and slot tables), and FP64 equilibria over the whole range of exponents."""
import numpy as np
import pytest

from paper_2303_10846_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def split_cavity(n=3, n_gh=5, half=False):
    """The cavity with every face of normal x (half: the interior ones) cut in two of half
    the area: the cells have eight (six to eight) faces, the closure is unchanged."""
    wl = I.cavity_workload(n=n, n_gh=n_gh)
    m = wl.mesh
    cut = np.abs(m.face_normal[:, 0]) > 0.5
    if half:
        cut &= m.face_cell[:, 1] >= 0
    o = np.concatenate([np.arange(m.n_face), np.nonzero(cut)[0]])
    second = np.arange(len(o)) >= m.n_face
    area, centre = m.face_area[o].copy(), m.face_center[o].copy()
    area[cut[o]] *= 0.5
    centre[cut[o], 1] += np.where(second[cut[o]], 0.25, -0.25) / n
    wl.mesh = I.Mesh(m.face_cell[o], m.face_normal[o], area, centre, m.cell_center, m.cell_volume, m.cell_colour)
    x = m.cell_center
    wl.prim0[:, 0] *= 1.0 + 0.1 * np.sin(5 * x[:, 0] + 3 * x[:, 1])
    wl.prim0[:, 4] *= 1.0 + 0.1 * np.cos(4 * x[:, 2])
    return wl


@pytest.mark.parametrize("prec,tol", [("fp64", 1e-10), ("mixed", 1e-5)])
@pytest.mark.parametrize("half", [False, True])
def test_cells_with_up_to_eight_faces_match_the_oracle(prec, tol, half):
    import oracle as O
    from paper_2303_10846_gb300.rykov import Solver
    wl = split_cavity(half=half)
    assert np.bincount(wl.mesh.face_cell[wl.mesh.face_cell >= 0].ravel()).max() == 8
    s, o = Solver(wl, prec), O.Oracle(wl)
    s.iterate(3)
    o.iterate(3)
    for name, buf in (("W", O.BUF_W), ("PHI", O.BUF_PHI), ("WT", O.BUF_WT)):
        a, b = s.debug_get(name), o.get(buf)
        assert np.abs(a.ravel() - b.ravel()).max() <= tol * np.abs(b).max(), name


def test_fp64_equilibrium_over_the_range_of_exponents():
    """Step 1 in FP64 against NumPy, element by element: velocities whose Maxwellian runs
    from 1 down past the smallest normal number.  The exponent, up to 690 where g > 1e-300,
    carries some ten roundings (|u|^2, the temperature from W, the scaling by log2 e, here
    and in NumPy) of 2^-53 each: 690 x 10 x 1.1e-16 < 1e-12."""
    from paper_2303_10846_gb300.rykov import Solver
    wl = I.cavity_workload(n=2, n_gh=4)
    r = np.linspace(0.0, 27.6, 1000)
    d = np.random.default_rng(5).normal(size=(1000, 3))
    u = r[:, None] * d / np.linalg.norm(d, axis=1)[:, None]
    wl.dvs = I.DVS(u=u, w=np.full(1000, 1e-3))
    s = Solver(wl, "fp64")
    phi = s.debug_get("PHI")
    # R = 1/2, T = 1, rho = 1, U = 0, q = 0: g = pi^-3/2 exp(-|u|^2), h = g/2
    g = np.pi ** -1.5 * np.exp(-(u * u).sum(1))
    normal = g > 1e-300
    for i in range(8):
        assert np.abs(phi[0, i, normal] / g[normal] - 1.0).max() < 1e-12
        assert np.abs(phi[1, i, normal] / (0.5 * g[normal]) - 1.0).max() < 1e-12
        assert np.abs(phi[0, i, ~normal] - g[~normal]).max() <= 1e-300


@pytest.mark.parametrize("prec,tol", [("fp64", 1e-10), ("mixed", 1e-5)])
@pytest.mark.parametrize("n_gh", [3, 5, 10, 17])
def test_velocity_counts_at_the_edges_of_the_forms(n_gh, prec, tol):
    """27 velocities (less than one step of a warp), 125 and 1,000 (ragged steps, one and
    several velocity blocks per cell), 4,913 (two warps per interior face): distributions,
    fields and wall sums against the oracle."""
    import oracle as O
    from paper_2303_10846_gb300.rykov import Solver
    wl = I.cavity_workload(n=3, n_gh=n_gh)
    x = wl.mesh.cell_center
    wl.prim0[:, 0] *= 1.0 + 0.1 * np.sin(5 * x[:, 0] + 3 * x[:, 1])
    wl.prim0[:, 4] *= 1.0 + 0.1 * np.cos(4 * x[:, 2])
    s, o = Solver(wl, prec), O.Oracle(wl)
    s.iterate(2)
    o.iterate(2)
    for name, buf in (("W", O.BUF_W), ("PHI", O.BUF_PHI), ("WT", O.BUF_WT), ("FACE", O.BUF_FACE)):
        a, b = s.debug_get(name), o.get(buf)
        assert np.abs(a.ravel() - b.ravel()).max() <= tol * np.abs(b).max(), name
    per, per_o = s.surface()[0], o.surface()[0]
    assert np.abs(per[:, 0] - per_o[:, 0]).max() <= tol * np.abs(per_o[:, 0]).max()
    assert not s.get_distribution()[:, :, wl.dvs.K:].any()


@pytest.mark.parametrize("prec,tol", [("fp64", 1e-10), ("mixed", 1e-5)])
@pytest.mark.parametrize("first_order", [False, True])
def test_adjoint_product_on_cells_with_eight_faces(first_order, prec, tol):
    """(dR/dX)^T v, (dR/dp)^T v and dJ/dX on the eight-faced cavity with an inflowing lid
    against autograd, FP64 to 1e-10 and mixed to 1e-5 of each block's largest entry (the
    tolerances of the adjoint's other tests)."""
    import torch
    from oracle.adjoint import HEAT, Steady
    from paper_2303_10846_gb300.rykov import Solver
    wl = split_cavity(n=2, n_gh=5)
    wl.bcs = [wl.bcs[0], I.BC(I.BC_FARFIELD, 1.05, (0.15, 0.02, -0.03), 1.1)]
    if first_order:
        wl.params.limiter = 2
    s = Solver(wl, prec)
    s.bind_adjoint(2)
    s.iterate(3)
    x = s.get_state()
    st = Steady(wl)
    v = np.random.default_rng(8).standard_normal(x.size)
    out, pp = s.vjp(v)
    ot, pt = st.vjp(torch.as_tensor(x), torch.as_tensor(v))
    J, g, dp = s.objective("heat")
    Jt, gt, dpt = st.objective_grad(torch.as_tensor(x), HEAT)
    n1, n2 = 2 * st.N * st.K, 2 * st.N * st.K + 6 * st.N
    for a, b in ((out, ot.numpy()), (g, gt.numpy())):
        for c in (slice(0, n1), slice(n1, n2), slice(n2, None)):
            assert np.abs(a[c] - b[c]).max() <= tol * max(np.abs(b[c]).max(), 1e-300)
    assert np.abs(pp - pt.numpy()).max() <= tol * np.abs(pt.numpy()).max()
    assert abs(J - Jt) <= tol * abs(Jt) and np.abs(dp - dpt.numpy()).max() <= tol * np.abs(dpt.numpy()).max()
    # in place: the output over the input
    w = torch.as_tensor(v, device="cuda")
    s._check(s.L.rk_vjp(s.h, w.data_ptr(), w.data_ptr(), None, 1))
    assert np.array_equal(w.cpu().numpy(), out)


@pytest.mark.parametrize("mesh", ["tetrahedra", "eight faces"])
@pytest.mark.parametrize("exponent", [20, 40, 70])
def test_mixed_reconstruction_is_homogeneous(mesh, exponent):
    """The limited reconstruction is homogeneous of degree 1 in the distribution and powers
    of two are exact, so scaling the distribution scales the interior face values bit for
    bit: by 2^-40 and 2^-70 the limiter's quotients are formed from rescaled operands."""
    import bench
    from paper_2303_10846_gb300 import rykov as RK
    wl = split_cavity() if mesh == "eight faces" else bench.dvs_sample(I.sphere_workload(h_wall=0.3, h_max=0.9), 23)
    wl.params.first_order_iters = 0
    s = RK.Solver(wl, "mixed")
    s.bind_adjoint(2)
    x = s.get_state()
    n1 = 2 * s.N * s.K
    x[:n1] = np.random.default_rng(3).uniform(0.5, 1.5, n1).astype(np.float32)
    interior = wl.mesh.face_cell[:, 1] >= 0
    out = []
    for e in (0, exponent):
        y = x.copy()
        y[:n1] *= 2.0 ** -e
        s.put_state(y)
        s.step(RK.STEP_RECON)
        out.append(s.debug_get("FACE")[:, interior] * 2.0 ** e)
    assert np.isfinite(out[0]).all() and np.abs(out[0] - 1.0).max() > 0.5
    assert np.array_equal(out[0], out[1])


@pytest.mark.parametrize("n,n_gh", [(6, 6), (8, 8)])
def test_settled_fp64_march_leaves_density_and_energy_where_they_are(n, n_gh):
    """A march that has settled: the macro solve's increment is zero to rounding, so W~ is W
    but for the last bit of a few cells.  The mean relative change of a step is then below a
    quarter of an ulp (2^-54); a solve whose own rounding is relative to W moves most cells
    by half an ulp or more."""
    from paper_2303_10846_gb300.rykov import Solver
    s = Solver(I.cavity_workload(n=n, n_gh=n_gh), "fp64")
    s.iterate(200)
    rho, energy = np.mean([s.iterate(5)[2][[0, 4]] for _ in range(20)], axis=0)
    assert rho <= 2.0 ** -54 and energy <= 2.0 ** -54, (rho, energy)


@pytest.mark.parametrize("a,b,product", [(200, 0, True), (0, 140, False), (160, 135, True), (-200, -140, False)])
def test_fp64_scheme_has_the_range_of_fp64(a, b, product):
    """Densities times 2^-a and velocities times 2^-b (the gas constant, the viscosity and
    the weights with them) scale the fields by powers of two: beyond the range of FP32 the
    march, the wall sums and the steady residual are the unscaled ones to rounding (1e-10,
    the tolerance of FP64 parity), and the adjoint product is finite (product: where the
    squared denominators of its limiter, products of four values of the distribution, are)."""
    import copy
    from paper_2303_10846_gb300.rykov import Solver
    from tests import workloads as TW
    base = TW.tiny_tet(n_gh=5, cfl_imp=20.0)
    wl = copy.deepcopy(base)
    r, c = 2.0 ** -a, 2.0 ** -b
    wl.prim0[:, 0] *= r
    wl.prim0[:, 1:4] *= c
    wl.dvs = I.DVS(u=base.dvs.u * c, w=base.dvs.w * c ** 3)
    wl.params.R *= c * c
    wl.params.mu_ref *= r * c
    wl.bcs = [I.BC(q.kind, q.rho * r, tuple(x * c for x in q.U), q.T) for q in base.bcs]
    wl.ref = dict(rho=r, U=tuple(x * c for x in base.ref["U"]), T=base.ref["T"])
    out = []
    for w in (base, wl):
        s = Solver(w, "fp64")
        s.bind_adjoint(2)
        s.iterate(3)
        W, q, _ = s.moments()
        per = s.surface()[0]
        R = s.steady_residual()[:2 * s.N * s.K].reshape(2, -1)
        v = s.vjp(np.ones(s.state_len))[0]
        out.append((W, q, per[:, :5], R, v))
    x, y = out
    scales = (np.array([r, r * c, r * c, r * c, r * c * c, r * c * c]), r * c ** 3,
              np.array([r * c * c] * 4 + [r * c ** 3]), np.array([[r / c ** 2], [r]]))
    for p, q, sc in zip(x, y, scales):
        z = q / sc
        assert np.abs(z - p).max() <= 1e-10 * np.abs(p).max()
    assert not product or np.isfinite(y[4]).all()


def test_mixed_padding_adds_nothing_beside_a_fast_velocity():
    """126 velocities (two of padding in the last group of four), one of them so fast that
    the cube of its speed, which the heat-flux terms form, is near the end of FP32's range
    (its Maxwellian is zero): the fields and macro fluxes are those of the FP64 context to the
    mixed tolerance."""
    from paper_2303_10846_gb300.rykov import Solver
    wl = I.cavity_workload(n=3, n_gh=5)
    x = wl.mesh.cell_center
    wl.prim0[:, 0] *= 1.0 + 0.1 * np.sin(5 * x[:, 0] + 3 * x[:, 1])
    fast = np.array([[2e12, 0.0, 0.0]])
    for at in (0, 125):
        u = np.insert(wl.dvs.u, at, fast, axis=0)
        w = np.insert(wl.dvs.w, at, 1e-3)
        wl2 = I.Workload(name="fast", mesh=wl.mesh, dvs=I.DVS(u=u, w=w), params=wl.params, bcs=wl.bcs,
                         prim0=wl.prim0, ref=wl.ref)
        m, d = Solver(wl2, "mixed"), Solver(wl2, "fp64")
        for s in (m, d):
            rc, n, res = s.iterate(2)
            assert rc == 0 and np.isfinite(res).all()
        for name in ("W", "MACRO_F"):
            a, b = m.debug_get(name), d.debug_get(name)
            assert np.abs(a - b).max() <= 1e-5 * np.abs(b).max(), name
        assert not m.get_distribution()[:, :, 126:].any()


def test_two_warps_per_interior_face():
    """5,832 velocities, beyond the line from which two warps share a face (one warp's rows
    end in the other's range): distributions, fields and face values against the oracle."""
    import oracle as O
    from paper_2303_10846_gb300.rykov import Solver
    wl = I.cavity_workload(n=3, n_gh=18)
    x = wl.mesh.cell_center
    wl.prim0[:, 0] *= 1.0 + 0.1 * np.sin(5 * x[:, 0] + 3 * x[:, 1])
    wl.prim0[:, 4] *= 1.0 + 0.1 * np.cos(4 * x[:, 2])
    s, o = Solver(wl, "mixed"), O.Oracle(wl)
    s.iterate(2)
    o.iterate(2)
    for name, buf in (("W", O.BUF_W), ("PHI", O.BUF_PHI), ("WT", O.BUF_WT), ("FACE", O.BUF_FACE)):
        a, b = s.debug_get(name), o.get(buf)
        assert np.abs(a.ravel() - b.ravel()).max() <= 1e-5 * np.abs(b).max(), name
