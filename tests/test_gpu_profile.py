"""oasis_profile: eager steps run the same kernels with and without it (the same bits), and
the families say which solves ran as one launch.  By sizes of rows and entries of K: every
solve resident; multigrid pressure above the limits of entries (box_44, 1.3 M) and between them
(box_42, 1.1 M); a float64 velocity solve above its limit of rows; one component and scalars;
forced shapes (separate kernels)."""
import numpy as np
import pytest

from test_gpu_resident import _lib, box3  # noqa: F401
from workloads import problems as WP

pytestmark = pytest.mark.gpu

STEPS = 2


@pytest.mark.parametrize("make,precision,opts,want", [
    (lambda: box3(9, 8, 10), 1, dict(pressure_pc=1), dict(bicg=1, cg=1)),
    (lambda: box3(9, 8, 10), 0, dict(pressure_pc=0), dict(bicg=1, cg=1)),
    (lambda: WP.taylor_green_2d(97), 0, dict(pressure_pc=1), dict(bicg=1, cg=1)),
    (lambda: box3(44, 43, 45), 1, dict(pressure_pc=1), dict(bicg=1, cg=0)),
    (lambda: box3(42, 41, 43), 0, dict(pressure_pc=1), dict(bicg=1, cg=0)),
    (lambda: box3(42, 41, 43), 1, dict(pressure_pc=1), dict(bicg=1, cg=1)),
    (lambda: box3(53, 52, 54), 0, dict(pressure_pc=1), dict(bicg=0, cg=0)),
    (lambda: WP.with_scalars(box3(14, 13, 12), ns=2), 1, dict(pressure_pc=1, velocity_update=1),
     dict(bicg=3, cg=1, mass=1)),
    (lambda: WP.with_scalars(box3(14, 13, 12), ns=2), 0, dict(pressure_pc=1, velocity_update=1, batch_rhs=0),
     dict(bicg=5, cg=1, mass=1)),
    (lambda: box3(14, 13, 12), 1, dict(pressure_pc=1, bicg_variant=1, spmv_variant=1), dict(bicg=0, cg=0)),
])
def test_profiled_steps_are_the_same_steps(make, precision, opts, want):
    from paper_1602_03643_gb300 import capi as c
    from paper_1602_03643_gb300.driver import IPCSRun
    out = []
    rtol = 1e-9 if precision else 1e-12
    pb = make()
    # one solver: two would differ in the shapes that their tuners choose
    run = IPCSRun(pb, precision=precision, rtol_u=rtol, rtol_p=rtol, use_graph=0, guess=1, **opts)
    try:
        for on in (False, True):
            c.oasis_set_fields(run.solver, pb.u_nm1, pb.u_nm2, pb.p, pb.t0, False, None)
            if run.ns:
                c.oasis_set_scalar_fields(run.solver, pb.scalars.c0, False, None)
            run.t = pb.t0
            c.oasis_profile(run.solver, on)
            run.step(STEPS)
            out.append(list(run.fields()) + ([run.scalar_fields()] if run.ns else []))
            fam = {f: c.oasis_profile_read(run.solver, f)[0] for f in c.PROF_FAMILIES}
    finally:
        run.close()
    for a, b in zip(*out):
        np.testing.assert_array_equal(a, b)
    assert fam["resident_bicg"] == STEPS * want["bicg"] and fam["resident_cg"] == STEPS * want["cg"]
    assert (fam["bicg_spmm"] > 0) == (want["bicg"] == 0) and (fam["pcg_spmv"] > 0) == (want["cg"] == 0)
    if "mass" in want:
        assert fam["mass"] == STEPS
