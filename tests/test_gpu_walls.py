"""Wall quantities from the wall faces alone: rk_surface and rk_aero reconstruct only the
cells at the walls; a debug context evaluates every face (the general path).  Both must
give the same bits, and a verification buffer read afterwards must be complete."""
import numpy as np
import pytest

from tests import workloads as TW

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("wl", [TW.tiny_cavity(2, 4), TW.tiny_cavity(4, 7), TW.tiny_tet(n_gh=5),
                                TW.tiny_tet(n_gh=7, lim=2)], ids=["cav2", "cav4_k343", "tet_k125", "tet_first"])
def test_wall_quantities_from_wall_faces_alone(wl, prec):
    from paper_2303_10846_gb300.rykov import Solver
    full, part = Solver(wl, prec, debug=True), Solver(wl, prec)
    for n in (0, 2):
        for s in (full, part):
            if n:
                s.iterate(n)
        a, b = full.surface(), part.surface()
        assert all(np.array_equal(x, y) for x, y in zip(a, b))
        assert np.array_equal(full.aero(), part.aero())
        assert np.array_equal(full.debug_get("FACE"), part.debug_get("FACE"))
        assert np.array_equal(full.debug_rows("FACE", [0, wl.mesh.n_face - 1]),
                              part.debug_rows("FACE", [0, wl.mesh.n_face - 1]))
    # the wall quantities leave the iteration as it is
    full.iterate(1)
    part.iterate(1)
    assert np.array_equal(full.moments()[0], part.moments()[0])


@pytest.mark.parametrize("debug", [False, True])
@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("wl", [TW.tiny_cavity(4, 5), TW.tiny_tet(n_gh=5)], ids=["cavity", "tet"])
def test_steps_with_wall_and_adjoint_calls_in_between(wl, prec, debug):
    """rk_surface, rk_aero and the FP32 adjoint use the face array as scratch: the steps
    around them, and the face values read after them, are those without the call (bit for
    bit: the same kernels on the same state)."""
    from paper_2303_10846_gb300 import rykov as RK
    steps = [RK.STEP_RECON, RK.STEP_FACES, RK.STEP_FLUXES, RK.STEP_MACRO, RK.STEP_MICRO]
    s = RK.Solver(wl, prec, debug=debug)
    s.bind_adjoint(2)
    s.iterate(2)
    x = s.get_state()
    v = np.random.default_rng(1).standard_normal(x.size)
    calls = {"surface": s.surface, "aero": s.aero, "vjp": lambda: s.vjp(v)}

    def run(call, at):
        s.put_state(x)
        for n, step in enumerate(steps):
            if n == at:
                calls[call]()
            s.step(step)
        return s.debug_get("FACE"), s.debug_get("MACRO_F"), s.moments()[0]

    s.put_state(x)
    for step in steps:
        s.step(step)
    ref = s.debug_get("FACE"), s.debug_get("MACRO_F"), s.moments()[0]
    for call in calls:
        for at in range(1, 5):
            for a, b in zip(run(call, at), ref):
                assert np.array_equal(a, b), (call, at)
    # read without a step in between: the finished faces of the present state
    s.put_state(x)
    s.surface()
    s.vjp(v)
    assert np.array_equal(s.debug_get("FACE"), ref[0])
    s.put_state(x)
    s.vjp(v)
    if prec == "mixed":
        assert np.array_equal(s.debug_rows("FACE", [0, wl.mesh.n_face - 1]), ref[0][:, [0, wl.mesh.n_face - 1]])
