"""A resident launch that the device refuses (its CTAs need more SMs at once than the
process or the stream may use): the passes run the streaming steps.

The library's objects are linked here against a stand-in for the CUDA runtime whose
device memory is host memory, whose kernels do nothing, and which can refuse
cooperative launches: the host path of a call is followed, without a GPU."""
import ctypes
import glob
import os
import subprocess

import numpy as np
import pytest

from paper_1406_1864_gb300 import _lib as L
from paper_1406_1864_gb300 import build as B

RUNTIME = r"""
#include <cstring>
#include <cuda.h>
#include <cuda_runtime_api.h>
static int g_refuse = 0, g_when = 0, g_refused = 0, g_cooperative = 0;
extern "C" {
// refuse: 0 nothing, 1 every cooperative launch, 2 all but the first `when` of them
void fake_set(int refuse, int when) { g_refuse = refuse, g_when = when, g_refused = g_cooperative = 0; }
int fake_refused() { return g_refused; }
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *c, const void *, void **)
{
    for (unsigned i = 0; i < c->numAttrs; ++i)
        if (c->attrs[i].id == cudaLaunchAttributeCooperative && c->attrs[i].val.cooperative) {
            const bool no = g_refuse == 1 || (g_refuse == 2 && g_cooperative >= g_when);
            ++g_cooperative;
            if (no) {
                ++g_refused;
                return cudaErrorCooperativeLaunchTooLarge;
            }
        }
    return cudaSuccess;
}
cudaError_t __cudaGetKernel(void **k, const void *) { *k = nullptr; return cudaSuccess; }
cudaError_t __cudaLaunchKernel(void *, dim3, dim3, void **, size_t, cudaStream_t) { return cudaSuccess; }
unsigned __cudaPushCallConfiguration(dim3, dim3, size_t, cudaStream_t) { return 0; }
cudaError_t __cudaPopCallConfiguration(dim3 *, dim3 *, size_t *, void *) { return cudaSuccess; }
void **__cudaRegisterFatBinary(void *) { static void *p; return &p; }
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterFunction(void **, const char *, char *, const char *, int, void *, void *, void *, void *, int *) {}
void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr, int) { *v = 152; return cudaSuccess; }
cudaError_t cudaGetDevice(int *d) { *d = 0; return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
const char *cudaGetErrorString(cudaError_t) { return "fake"; }
cudaError_t cudaGetSymbolAddress(void **p, const void *) { *p = nullptr; return cudaErrorInvalidSymbol; }
cudaError_t cudaFuncSetAttribute(const void *, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessor(int *n, const void *, int, size_t) { *n = 4; return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int *n, const void *, int, size_t, unsigned)
{ *n = 4; return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind, cudaStream_t) { memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemsetAsync(void *d, int v, size_t n, cudaStream_t) { memset(d, v, n); return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t *e) { *e = (cudaEvent_t)1; return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { *e = (cudaEvent_t)1; return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t, cudaEvent_t) { *ms = 0; return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventRecordWithFlags(cudaEvent_t, cudaStream_t, unsigned) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t *g) { *g = (cudaGraph_t)1; return cudaSuccess; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *x, cudaGraph_t, unsigned long long) { *x = (cudaGraphExec_t)1; return cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
static CUresult encode(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *, const cuuint64_t *,
                       const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                       CUtensorMapL2promotion, CUtensorMapFloatOOBfill) { return CUDA_SUCCESS; }
cudaError_t cudaGetDriverEntryPointByVersion(const char *name, void **f, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult *q)
{
    const bool tm = strcmp(name, "cuTensorMapEncodeTiled") == 0;
    *f = tm ? (void *)encode : nullptr;
    if (q) *q = tm ? cudaDriverEntryPointSuccess : cudaDriverEntryPointSymbolNotFound;
    return cudaSuccess;
}
}
"""

NZ, NX, NS, NT = 37, 83, 3, 21


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    B.build()
    objs = sorted(glob.glob(os.path.join(B.BUILD, "*.o")))
    if len(objs) != len(B.sources()):
        B.build(force=True)
        objs = sorted(glob.glob(os.path.join(B.BUILD, "*.o")))
    d = tmp_path_factory.mktemp("refused")
    (d / "runtime.cpp").write_text(RUNTIME)
    so = str(d / "libfwi_fake.so")
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    subprocess.check_call(["g++", "-std=c++17", "-shared", "-fPIC", f"-I{cuda}/include", str(d / "runtime.cpp")] + objs +
                          ["-Wl,-Bsymbolic", "-Wl,-z,defs", "-lpthread", "-ldl", "-o", so])
    h = ctypes.CDLL(so)
    for name, args in L._SIGS.items():
        getattr(h, name).argtypes = args
    h.fwi_last_error.restype = ctypes.c_char_p
    assert h.fwi_profile_enable(1) == L.FWI_OK
    return h


class Problem:
    def __init__(self):
        src = np.zeros((NS, 3), np.int32)
        src[:, 2] = [0, 40, NX - 1]
        rec = np.zeros((NS, NX, 3), np.int32)
        rec[:, :, 0], rec[:, :, 2] = 1, np.arange(NX)
        self.keep = [src, rec, np.zeros((NS, NT), np.float32)]
        self.grid = L.FwiGrid(2, NZ, 1, NX, 10.0, 1e-3, NT, 7, 3000.0, 0.05)
        self.geom = L.FwiGeometry(NS, NX, src.ctypes.data, rec.ctypes.data, self.keep[2].ctypes.data)
        self.opts = L.FwiOptions(0, 0, 3, 2, 1e-3)
        self.v = np.full((NZ, NX), 2500.0, np.float32)
        self.seis = np.zeros((NS, NT, NX), np.float32)
        self.out = np.zeros((8, NZ, NX), np.float32)
        self.misfit = np.zeros(1)


def buffer(n):
    raw = np.zeros(n + 256, np.uint8)
    off = -raw.ctypes.data % 256
    return raw[off:off + n]


def forward(lib, save):
    p, n = Problem(), ctypes.c_size_t(0)
    assert lib.fwi_workspace_bytes(p.grid, p.geom, p.opts, L.FWI_OP_FORWARD_SAVE if save else L.FWI_OP_FORWARD, n) == L.FWI_OK
    ws = buffer(n.value)
    st = lib.fwi_forward(p.grid, p.geom, p.opts, p.v.ctypes.data, p.seis.ctypes.data, save, ws.ctypes.data, n, None)
    return st, ws


def gradient(lib, models=1, record=False):
    p, n = Problem(), ctypes.c_size_t(0)
    grids, geoms = (L.FwiGrid * models)(*[p.grid] * models), (L.FwiGeometry * models)(*[p.geom] * models)
    assert lib.fwi_workspace_preferred_bytes(models, grids, geoms, p.opts, L.FWI_OP_GRADIENT, n) == L.FWI_OK
    ws = buffer(n.value)

    def each(x):
        return (ctypes.c_void_p * models)(*[x.ctypes.data] * models)

    if models == 1 and not record:
        st = lib.fwi_adjoint_gradient(p.grid, p.geom, p.opts, p.v.ctypes.data, p.seis.ctypes.data, p.out[0].ctypes.data,
                                      p.out[1].ctypes.data, p.misfit.ctypes.data, p.out[2].ctypes.data,
                                      p.out[3].ctypes.data, ws.ctypes.data, n, None)
        return st, ws
    mis = np.zeros(models)
    args = (models, grids, geoms, p.opts, each(p.v), each(p.seis), each(p.out[0]), each(p.out[1]), mis.ctypes.data,
            each(p.out[2]), each(p.out[3]), ws.ctypes.data, n)
    if not record:
        return lib.fwi_batch_gradient(*args, None), ws
    ex = ctypes.c_void_p(0)
    st = lib.fwi_exec_gradient_create(*args, ctypes.c_void_p(64), ctypes.byref(ex))
    if st == L.FWI_OK:
        st = lib.fwi_exec_run(ex, ctypes.c_void_p(64))
        assert lib.fwi_exec_destroy(ex) == L.FWI_OK
    return st, ws


def launches(lib):
    t = L.FwiPhaseTimes()
    assert lib.fwi_profile_last(ctypes.byref(t)) == L.FWI_OK
    return t.forward_launches, t.adjoint_launches


CALLS = {"forward": lambda lib: forward(lib, 0), "forward_save": lambda lib: forward(lib, 1), "gradient": gradient,
         "batch": lambda lib: gradient(lib, 2), "graph": lambda lib: gradient(lib, 1, True)}


@pytest.mark.parametrize("name", list(CALLS))
def test_refused_resident_launches_run_the_streaming_steps(lib, name):
    """Status, launches and what the call leaves in its workspace (the receiver tables
    of the streaming tilings among it) are those of a call whose steps are pinned."""
    p, back = Problem(), 0 if name.startswith("forward") else NT - 1
    assert lib.fwi_autotune_reset() == L.FWI_OK
    lib.fake_set(0, 0)
    assert CALLS[name](lib)[0] == L.FWI_OK
    resident = launches(lib)
    assert resident[0] < NT and resident[1] < max(1, back)
    lib.fake_set(1, 0)
    st, ws = CALLS[name](lib)
    assert st == L.FWI_OK, lib.fwi_last_error()
    assert lib.fake_refused() > 0 and launches(lib) == (NT, back)
    lib.fake_set(0, 0)
    for hmax, variant in ((-1, 0), (3, 2)):
        choice = (ctypes.c_int * 4)(3 if hmax < 0 else variant, 8 if hmax < 0 else 16, 1, 8)
        o = L.FwiOptions(0, 0, hmax, 1, 1e-3)
        assert lib.fwi_autotune_set(p.grid, p.geom, o, choice) == L.FWI_OK
    st, pinned = CALLS[name](lib)
    assert lib.fwi_autotune_reset() == L.FWI_OK
    assert st == L.FWI_OK and launches(lib) == (NT, back)
    if name != "forward_save":  # (which leaves the tables of the adjoint pass as planned)
        assert np.array_equal(ws[:len(pinned)], pinned)


@pytest.mark.parametrize("name,first", [("gradient", 1), ("batch", 1), ("batch", 3)])
def test_a_later_launch_is_refused(lib, name, first):
    """The forward pass has run resident when the adjoint one, or another model of a
    batch, is refused."""
    assert lib.fwi_autotune_reset() == L.FWI_OK
    lib.fake_set(2, first)
    st, _ = CALLS[name](lib)
    assert st == L.FWI_OK, lib.fwi_last_error()
    assert lib.fake_refused() == 1 or name == "batch"
    assert launches(lib)[1] >= NT - 1
