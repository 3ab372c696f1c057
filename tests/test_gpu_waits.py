"""The meetings of blocks inside one launch give up after a limit.

With a limit of one clock cycle a block that has to wait for another leaves its launch; the
others then wait in vain for it, and every launch ends by itself.  The call must say
OASIS_EWAIT.  With the usual limit again, the same solver gives the bits of one that was
never disturbed: the meeting memory was left clean.
"""
import numpy as np
import pytest

from test_gpu_resident import _lib, box3  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,graph,opts", [
    (1, 0, dict(pressure_pc=1, velocity_update=1)), (1, 1, dict(pressure_pc=1, velocity_update=1)),
    (0, 0, dict(pressure_pc=0)), (0, 1, dict(pressure_pc=0)),
    # separate kernels: the meetings are those of the V-cycle's shared launch
    (1, 1, dict(pressure_pc=1, bicg_variant=1, spmv_variant=1)),
    (0, 1, dict(pressure_pc=1, bicg_variant=1, spmv_variant=1))])
def test_steps_report_a_wait_that_ran_out(precision, graph, opts):
    from paper_1602_03643_gb300 import capi as c
    from paper_1602_03643_gb300.driver import IPCSRun
    rtol = 1e-9 if precision else 1e-12
    run = IPCSRun(box3(30, 30, 31), precision=precision, rtol_u=rtol, rtol_p=rtol, use_graph=graph, guess=0, **opts)
    try:
        pb = run.pb
        run.step()
        want = run.fields()
        c.oasis_set_wait_limit(run.solver, 1)
        with pytest.raises(c.OasisError) as e:
            run.step()
        assert e.value.code == c.OASIS_EWAIT
        c.oasis_set_wait_limit(run.solver, 0)
        c.oasis_set_fields(run.solver, pb.u_nm1, pb.u_nm2, pb.p, pb.t0, False, None)
        run.t = pb.t0
        run.step()
        for a, b in zip(run.fields(), want):
            np.testing.assert_array_equal(a, b)
        with pytest.raises(c.OasisError) as e:
            c.oasis_set_wait_limit(run.solver, -1)
        assert e.value.code == c.OASIS_EINVAL
    finally:
        run.close()


@pytest.mark.parametrize("precision", [0, 1])
def test_amg_apply_reports_a_wait_that_ran_out(precision):
    import torch
    from paper_1602_03643_gb300 import capi as c
    from paper_1602_03643_gb300.driver import IPCSRun
    run = IPCSRun(box3(30, 30, 31), precision=precision, pressure_pc=1)
    try:
        r = torch.randn(run.n, device="cuda", dtype=torch.float32 if precision else torch.float64)
        out = [torch.empty_like(r) for _ in range(3)]
        c.oasis_amg_apply(run.solver, r, out[0])
        c.oasis_set_wait_limit(run.solver, 1)
        with pytest.raises(c.OasisError) as e:
            c.oasis_amg_apply(run.solver, r, out[1])
        assert e.value.code == c.OASIS_EWAIT
        c.oasis_set_wait_limit(run.solver, 0)
        c.oasis_amg_apply(run.solver, r, out[2])
        assert torch.equal(out[0], out[2])
    finally:
        run.close()
