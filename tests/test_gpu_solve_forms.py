"""Error statuses and options of the linear solves in both of their forms: one launch
(forced = 0 on these sizes) and separate kernels (forced = 1).

Sizes of the options: 2D with two lanes per row, 3D with one lane per row (mixed) and a
matrix too large for shared memory (float64, from ~80,000 rows).  Bounds: those of
test_gpu_resident.py.
"""
import numpy as np
import pytest

from test_gpu_resident import _lib, box3, relerr  # noqa: F401
from workloads import problems as WP

pytestmark = pytest.mark.gpu


def launched_as_one(run):
    from paper_1602_03643_gb300 import capi as c
    return {f: c.oasis_profile_read(run.solver, f)[0] for f in ("resident_bicg", "resident_cg", "mass")}


@pytest.mark.parametrize("graph,forced", [(0, 0), (1, 0), (1, 1)])
@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("opts", [
    dict(pressure_pc=0, max_it_p=2), dict(pressure_pc=1, max_it_p=1), dict(pressure_pc=1, max_it_u=1),
    dict(pressure_pc=1, max_it_u=1, batch_rhs=0)])
def test_notconv(opts, precision, graph, forced):
    from paper_1602_03643_gb300 import capi as c
    from paper_1602_03643_gb300.driver import IPCSRun
    run = IPCSRun(WP.taylor_green_3d(9), precision=precision, rtol_u=1e-9, rtol_p=1e-9, use_graph=graph,
                  bicg_variant=forced, spmv_variant=forced, **opts)
    try:
        with pytest.raises(c.OasisError) as e:
            run.step()
        assert e.value.code == c.OASIS_ENOTCONV
    finally:
        run.close()


@pytest.mark.parametrize("graph,forced", [(0, 0), (1, 0), (1, 1)])
@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("pc", [0, 1])
def test_nan(pc, precision, graph, forced):
    from paper_1602_03643_gb300 import capi as c
    from paper_1602_03643_gb300.driver import IPCSRun
    pb = WP.taylor_green_3d(9)
    pb.u_nm1 = pb.u_nm1.copy()
    pb.u_nm1[0, 100] = np.nan
    run = IPCSRun(pb, precision=precision, rtol_u=1e-9, rtol_p=1e-9, use_graph=graph, pressure_pc=pc,
                  bicg_variant=forced, spmv_variant=forced, max_it_u=300, max_it_p=300)
    try:
        with pytest.raises(c.OasisError) as e:
            run.step()
        assert e.value.code in (c.OASIS_ENAN, c.OASIS_ENOTCONV)
    finally:
        run.close()


MESHES = {"square_190": lambda: WP.taylor_green_2d(190), "box_38": lambda: box3(38, 37, 39),
          "box_44": lambda: box3(44, 43, 45)}


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("name", list(MESHES))
@pytest.mark.parametrize("opts", [dict(batch_rhs=0), dict(velocity_update=1), dict(scalars=2)])
def test_options_in_both_forms(opts, name, precision):
    from paper_1602_03643_gb300 import capi as c
    from paper_1602_03643_gb300.driver import IPCSRun
    opts = dict(opts)
    pb = MESHES[name]()
    ns = opts.pop("scalars", 0)
    if ns:
        pb = WP.with_scalars(pb, ns=ns)
    rtol = 1e-12 if precision == 0 else 1e-9
    out = []
    for forced in (0, 1):
        # eager steps tell what they launched
        run = IPCSRun(pb, precision=precision, rtol_u=rtol, rtol_p=rtol, use_graph=forced, pressure_pc=1, guess=1,
                      bicg_variant=forced, spmv_variant=forced, **opts)
        try:
            c.oasis_profile(run.solver, True)
            st = run.step(2)
            assert st.status == 0
            if not forced:
                one = launched_as_one(run)
                assert one["resident_bicg"] == 2 * (ns + (pb.mesh.dim if opts.get("batch_rhs") == 0 else 1))
                assert one["mass"] == (2 if opts.get("velocity_update") else 0)
                assert one["resident_cg"] == (0 if name == "box_44" else 2)
            out.append(list(run.fields()[:2]) + ([run.scalar_fields()] if run.ns else []))
        finally:
            run.close()
    for x, y in zip(*out):
        assert relerr(x, y) < (1e-9 if precision == 0 else 1e-6)
