"""Resident launches need all their blocks on the GPU at once.  On a stream that may use only some of
the SMs (a green context) a lattice whose grid is larger steps with a launch per pass instead, and
one whose grid fits stays resident; results as on the whole GPU."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

from tests import inputs

pytestmark = pytest.mark.gpu

HELPER = r"""
#include <cuda.h>
// A stream on `sms` SMs or a few more of device 0, by a green context that lives with the process.
extern "C" int partial_stream(unsigned sms, CUstream* stream, unsigned* got)
{
    CUdevice dev;
    CUdevResource all, part, rest;
    CUdevResourceDesc desc;
    CUgreenCtx ctx;
    unsigned n = 1;
    CUresult r = cuInit(0);
    if (r == CUDA_SUCCESS) r = cuDeviceGet(&dev, 0);
    if (r == CUDA_SUCCESS) r = cuDeviceGetDevResource(dev, &all, CU_DEV_RESOURCE_TYPE_SM);
    if (r == CUDA_SUCCESS) r = cuDevSmResourceSplitByCount(&part, &n, &all, &rest, 0, sms);
    if (r == CUDA_SUCCESS) r = cuDevResourceGenerateDesc(&desc, &part, 1);
    if (r == CUDA_SUCCESS) r = cuGreenCtxCreate(&ctx, desc, dev, CU_GREEN_CTX_DEFAULT_STREAM);
    if (r == CUDA_SUCCESS) r = cuGreenCtxStreamCreate(stream, ctx, CU_STREAM_NON_BLOCKING, 0);
    *got = part.sm.smCount;
    return r;
}
"""


@pytest.fixture(scope="module")
def cl():
    from paper_2607_24978_gb300 import build_ext, cl as mod
    build_ext.build()
    mod.lib()
    return mod


@pytest.fixture(scope="module")
def few_sms(cl, tmp_path_factory):
    d = tmp_path_factory.mktemp("green")
    (d / "green.cu").write_text(HELPER)
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    subprocess.run([os.path.join(cuda, "bin", "nvcc"), "-shared", "-Xcompiler", "-fPIC", str(d / "green.cu"), "-o",
                    str(d / "green.so"), "-L" + os.path.join(cuda, "lib64", "stubs"), "-lcuda"], check=True)
    stream, got = C.c_void_p(), C.c_uint()
    r = C.CDLL(str(d / "green.so")).partial_stream(C.c_uint(16), C.byref(stream), C.byref(got))
    if r != 0:
        pytest.skip("no green context here (CUresult %d)" % r)
    assert 0 < got.value <= 32
    return stream.value


# 32^3: 64 blocks; 48^3: more; 8^3: a few blocks, which fit
@pytest.mark.parametrize("N,nf,prec", [(32, 1, 1), (48, 2, 0), (8, 1, 0)])
def test_steps_on_some_of_the_sms(cl, few_sms, N, nf, prec):
    phi, pi = inputs.scalar_state(N, nf, seed=N, fbar=(1.0, 0.1), amp=0.05, pamp=0.05)
    dtype = np.float64 if prec == 0 else np.float32
    out = []
    for stream in (None, few_sms):
        with cl.Lattice(N, 0.4 * N, nf, prec, cl.CL_INT_YOSHIDA4, expansion=True, alpha=0.5, kappa=0.2, dt=0.005,
                        stream=stream) as g:
            g.cl_set_potential(cl.CL_POT_POLY, [0.5, 1.0, 0.2 if nf == 2 else 0.0, 0.4 if nf == 2 else 0.0,
                                                3.0 if nf == 2 else 0.0])
            for f in range(nf):
                g.cl_set_state(cl.CL_FIELD_PHI0 + f, phi[f].astype(dtype))
                g.cl_set_state(cl.CL_FIELD_PI0 + f, pi[f].astype(dtype))
            g.cl_set_scalars(1.0, 0.3, 0.0)
            counts = []
            for n in (2, 3):
                g.cl_step(n)
                counts.append(g.cl_last_launch_count())
            out.append((counts, g.cl_energies(), [g.cl_get_state(cl.CL_FIELD_PHI0 + f) for f in range(nf)]))
    a, b = out
    assert a[0] == b[0] == [7, 9]
    tol = 1e-12 if prec == 0 else 1e-6  # as between the two forms on the whole GPU
    for x, y in zip(a[2], b[2]):
        assert np.max(np.abs(x - y)) <= tol * np.max(np.abs(x))
    for k in ("t", "a", "adot", "rho"):
        assert b[1][k] == pytest.approx(a[1][k], rel=max(tol, 1e-11) if prec == 0 else 1e-7), k
    assert a[1]["step"] == b[1]["step"] == 5
