"""Steps on a stream that has only a few of the device's multiprocessors (a green context):
launches that need all their CTAs on the device at once are refused there, and the
kernels that need no such launch take the step.  The same problem on an ordinary stream
is the reference; the solves are those of other kernels, so the fields agree to the
tolerance of the solves."""
import ctypes
import subprocess

import pytest

torch = pytest.importorskip("torch")

from paper_2204_13254_gb300 import dd as D
from paper_2204_13254_gb300 import workloads as W

pytestmark = pytest.mark.gpu

HELPER = r"""
#include <cuda.h>
static CUgreenCtx ctx;
// A stream on `sms` multiprocessors; returns how many it has, or minus the error.
int open_part(unsigned sms, CUstream* stream) {
    CUdevice dev;
    CUdevResource all, part;
    CUdevResourceDesc desc;
    unsigned groups = 1;
    CUresult e = cuDeviceGet(&dev, 0);
    if (!e) e = cuDeviceGetDevResource(dev, &all, CU_DEV_RESOURCE_TYPE_SM);
    if (!e) e = cuDevSmResourceSplitByCount(&part, &groups, &all, 0, 0, sms);
    if (!e) e = cuDevResourceGenerateDesc(&desc, &part, 1);
    if (!e) e = cuGreenCtxCreate(&ctx, desc, dev, CU_GREEN_CTX_DEFAULT_STREAM);
    if (!e) e = cuGreenCtxStreamCreate(stream, ctx, CU_STREAM_NON_BLOCKING, 0);
    return e ? -(int)e : (int)part.sm.smCount;
}
int close_part(CUstream stream) {
    CUresult e = cuStreamSynchronize(stream);
    if (!e) e = cuStreamDestroy(stream);
    return (int)(e ? e : cuGreenCtxDestroy(ctx));
}
"""


@pytest.fixture(scope="module")
def part(tmp_path_factory):
    """(stream, multiprocessors)"""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.zeros(1, device="cuda")
    ctypes.CDLL("libcuda.so.1", mode=ctypes.RTLD_GLOBAL)
    src = tmp_path_factory.mktemp("part") / "part.c"
    src.write_text(HELPER)
    so = src.with_suffix(".so")
    subprocess.run(["gcc", "-shared", "-fPIC", "-I/usr/local/cuda/include", str(src), "-o", str(so)], check=True)
    lib = ctypes.CDLL(str(so))
    lib.close_part.argtypes = [ctypes.c_void_p]
    stream = ctypes.c_void_p()
    n = lib.open_part(8, ctypes.byref(stream))
    if n <= 0:
        pytest.skip(f"no green context (driver error {-n})")
    yield torch.cuda.ExternalStream(stream.value), n
    assert lib.close_part(stream) == 0


GMRES, CG = D.DD_SOLVER_COUPLED_GMRES, D.DD_SOLVER_SCHUR_CG


@pytest.mark.parametrize("n, k, prec, solver", [(16, 4, D.DD_FP64, GMRES), (16, 4, D.DD_FP64, CG), (12, 6, D.DD_FP64, CG),
                                                (12, 6, D.DD_MIXED, CG), (12, 6, D.DD_MIXED, GMRES)])
def test_step_on_a_part_of_the_device(part, n, k, prec, solver):
    """One-kernel Arnoldi and CG steps (64 subdomains), one-kernel solves (216 subdomains)."""
    stream, sms = part
    w = W.box(n, n, n, k, k, k)
    mixed = prec == D.DD_MIXED
    fs = D.FieldSolver(w.xyz, w.tets, w.part, w.n_sub, params=D.make_params(
        precision=prec, solver=solver, tol=1e-5 if mixed else 1e-13, refine_tol=1e-11, max_refine=8, max_it=2000)).bind()
    fs.factor(0.46 / n)
    ctas = fs.n_lambda // 512 if k == 4 else w.n_sub     # of the launches that have to be refused
    assert ctas > sms
    src = torch.randn(fs.n_dof, dtype=torch.float64, generator=torch.Generator().manual_seed(2)).cuda()
    out = [torch.empty_like(src) for _ in range(4)]
    zero = torch.zeros_like(src)
    for q, s in enumerate((None, stream)):
        fs.set_state(zero, zero, 0)
        for step in range(2):
            torch.cuda.synchronize()
            D.dd_step(fs.h, src, out[2 * q + step], stats=True, stream=s)
            if s is not None:
                s.synchronize()
    for a, b in zip(out[:2], out[2:]):
        assert torch.linalg.norm(a - b) <= 1e-9 * torch.linalg.norm(a)
    fs.close()
