"""Solves on a device that refuses the resident solves' cooperative launches.

The refusal is made on the host: a preloaded library answers the runtime's questions (no
cooperative launches; MPS in use; no block of a kernel fits) and fails every cooperative
launch with the error that such a device gives.  Steps must then run as separate kernels,
and agree with the same steps without the library to the bounds between the resident and
the separate solves (test_gpu_resident.py).
"""
import os
import shutil
import subprocess
import sys

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

FAKE = r"""
#define _GNU_SOURCE
#include <dlfcn.h>
#include <stdlib.h>
#include <string.h>
#include <cuda_runtime_api.h>

static const char* fake(void) { const char* f = getenv("FAKE_DEVICE"); return f ? f : ""; }

cudaError_t cudaDeviceGetAttribute(int* v, enum cudaDeviceAttr what, int dev) {
    cudaError_t (*real)(int*, enum cudaDeviceAttr, int) = dlsym(RTLD_NEXT, "cudaDeviceGetAttribute");
    if (what == cudaDevAttrCooperativeLaunch && !strcmp(fake(), "no_cooperative")) { *v = 0; return cudaSuccess; }
    if (what == cudaDevAttrMpsEnabled && !strcmp(fake(), "mps")) { *v = 1; return cudaSuccess; }
    return real(v, what, dev);
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void* fn, int block, size_t smem,
                                                                   unsigned flags) {
    cudaError_t (*real)(int*, const void*, int, size_t, unsigned) =
        dlsym(RTLD_NEXT, "cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags");
    // the separate kernels have 256 threads at most, the launch of a solve more from 38,913 rows on
    if (block > 256 && !strcmp(fake(), "no_room")) { *n = 0; return cudaSuccess; }
    return real(n, fn, block, smem, flags);
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* fn, void** args) {
    cudaError_t (*real)(const cudaLaunchConfig_t*, const void*, void**) = dlsym(RTLD_NEXT, "cudaLaunchKernelExC");
    for (unsigned k = 0; *fake() && k < c->numAttrs; ++k)
        if (c->attrs[k].id == cudaLaunchAttributeCooperative && c->attrs[k].val.cooperative)
            return cudaErrorCooperativeLaunchTooLarge;
    return real(c, fn, args);
}
"""

RUN = r"""
import sys
import numpy as np
from test_gpu_resident import box3
from paper_1602_03643_gb300.driver import IPCSRun
from workloads import problems as WP
prec, pc, graph, forced, scalars, update, big = map(int, sys.argv[2:])
pb = box3(*((14, 13, 12), (30, 30, 31), (34, 33, 35))[big])
if scalars:
    pb = WP.with_scalars(pb, ns=scalars)
rtol = 1e-9 if prec else 1e-12
run = IPCSRun(pb, precision=prec, rtol_u=rtol, rtol_p=rtol, use_graph=graph, pressure_pc=pc, guess=1,
              bicg_variant=forced, spmv_variant=forced, velocity_update=update)
st = run.step(2)
assert st.status == 0
u, p, _ = run.fields()
np.savez(sys.argv[1], u=u, p=p, c=run.scalar_fields() if run.ns else np.zeros(1))
run.close()
"""


@pytest.fixture(scope="module")
def fake_device(tmp_path_factory):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    cc = shutil.which("gcc")
    if not cc:
        pytest.skip("no C compiler")
    from paper_1602_03643_gb300 import build
    build.build()
    at = tmp_path_factory.mktemp("fake")
    src, lib = at / "fake.c", at / "fake.so"
    src.write_text(FAKE)
    include = os.path.join(os.path.dirname(os.path.dirname(build.nvcc())), "include")
    subprocess.run([cc, "-shared", "-fPIC", "-I", include, str(src), "-o", str(lib), "-ldl"], check=True)
    return at, lib


@pytest.mark.parametrize("fake,prec,pc,graph,forced,scalars,update,big", [
    ("no_cooperative", 1, 1, 1, 0, 2, 1, 0), ("no_cooperative", 0, 0, 0, 0, 0, 0, 0), ("no_room", 1, 0, 1, 0, 0, 0, 2),
    # the V-cycle's shared launch, inside and outside of a conditional body
    ("mps", 1, 1, 1, 1, 0, 0, 1), ("mps", 0, 1, 0, 1, 0, 0, 1)])
def test_separate_kernels_where_cooperative_launches_are_refused(fake_device, fake, prec, pc, graph, forced, scalars,
                                                                 update, big):
    at, lib = fake_device
    out = []
    for name in ("", fake):
        env = dict(os.environ, PYTHONPATH=os.pathsep.join([ROOT, os.path.join(ROOT, "tests")]), FAKE_DEVICE=name,
                   LD_PRELOAD=str(lib))
        res = at / f"out{name}.npz"
        r = subprocess.run([sys.executable, "-c", RUN, str(res)] + [str(v) for v in
                           (prec, pc, graph, forced, scalars, update, big)], env=env, cwd=ROOT, capture_output=True,
                           text=True, timeout=120)
        assert r.returncode == 0, r.stderr[-2000:]
        out.append(np.load(res))
    for k, tol in (("u", 1e-6 if prec else 1e-9), ("p", 1e-6 if prec else 1e-9), ("c", 1e-6 if prec else 1e-9)):
        a, b = out[0][k], out[1][k]
        assert np.linalg.norm(a - b) <= tol * max(np.linalg.norm(a), 1e-300), k
