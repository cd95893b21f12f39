"""Which launches lbm13_step and lbm13_plan_step make, and what they do when a CUDA
call fails: lbm13_api.cu compiled with the host compiler against a stand-in for the
CUDA runtime, whose memory is the host's, whose calls fail when told to and whose
launches write a log (s: a step, g: a graph of 32, R<n>: n steps from shared memory,
M<n>: n steps with grid barriers, b: a batched step, P<n>: a plan's n steps from
shared memory)."""
import ctypes as C
import os
import shutil
import subprocess

import numpy as np
import pytest

from paper_1401_0188_gb300 import lbm13 as B
from paper_1401_0188_gb300 import pstar, rest_temperature
from paper_1401_0188_gb300 import workloads as W

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1401_0188_gb300", "csrc")
CUDA_INC = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")
AUTO, OFF, ON = 0, 1, 2
FP64, FP32 = 0, 1

FAKE = r"""
#include <cstdlib>
#include <cstring>
#include <map>
#include <set>
#include <string>
#include "lbm13_internal.h"
#include "lbm13_tma.h"
#include "lbm13_pair.h"
#include "lbm13_resident.h"
using namespace lbm13;

// what the stand-in does: the n-th next memset, allocation or resident launch fails;
// attributes; whether the lattice's stream, or another one of the process, is captured
extern "C" {
int fake_fail_memset = 0, fake_fail_malloc = 0, fake_fail_resident = 0, fake_cooperative = 1, fake_capturing = 0,
    fake_blocks_per_sm = 1, fake_other_capture = 0;
}
static std::string g_log;
static std::map<void *, size_t> g_mem;
static std::set<void *> g_own;
static bool g_capture = false, g_relaxed = false;
extern "C" const char *fake_log() { return g_log.c_str(); }
extern "C" void fake_clear() { g_log.clear(); }
extern "C" int fake_allocations() { return int(g_mem.size()); }
static bool hit(int &n) { return n > 0 && --n == 0; }

extern "C" int fake_encode() { return 0; }  // cuTensorMapEncodeTiled
extern "C" {
cudaError_t cudaMalloc(void **p, size_t n)
{
    if (hit(fake_fail_malloc)) return cudaErrorMemoryAllocation;
    if (fake_other_capture && !g_relaxed) return cudaErrorStreamCaptureUnsupported;
    *p = std::malloc(n);
    std::memset(*p, 0xa5, n);  // as memory comes
    g_mem[*p] = n;
    return cudaSuccess;
}
cudaError_t cudaFree(void *p)
{
    g_mem.erase(p);
    std::free(p);
    return cudaSuccess;
}
cudaError_t cudaMemset(void *p, int v, size_t n) { std::memset(p, v, n); return cudaSuccess; }
cudaError_t cudaMemsetAsync(void *p, int v, size_t n, cudaStream_t)
{
    if (hit(fake_fail_memset)) return cudaErrorInvalidValue;
    std::memset(p, v, n);
    return cudaSuccess;
}
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, cudaMemcpyKind) { std::memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind, cudaStream_t) { std::memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemcpy2DAsync(void *, size_t, const void *, size_t, size_t, size_t, cudaMemcpyKind, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGetDevice(int *d) { *d = 0; return cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaGetDeviceProperties(cudaDeviceProp *p, int) { std::memset(p, 0, sizeof *p); p->multiProcessorCount = 152; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr a, int)
{
    *v = a == cudaDevAttrCooperativeLaunch ? fake_cooperative : a == cudaDevAttrMultiProcessorCount ? 152 : 0;
    return cudaSuccess;
}
cudaError_t cudaDeviceSynchronize() { return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
const char *cudaGetErrorString(cudaError_t e) { return e == cudaSuccess ? "no error" : "an error"; }
cudaError_t cudaEventCreate(cudaEvent_t *e) { *e = reinterpret_cast<cudaEvent_t>(std::malloc(1)); return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t e) { std::free(e); return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *t, cudaEvent_t, cudaEvent_t) { *t = 1.0f; return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) { *s = reinterpret_cast<cudaStream_t>(std::malloc(1)); return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t s) { std::free(s); return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus *c)
{
    *c = fake_capturing ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
    return cudaSuccess;
}
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { g_capture = true; return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t *g) { g_capture = false; *g = reinterpret_cast<cudaGraph_t>(std::malloc(1)); return cudaSuccess; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *x, cudaGraph_t, unsigned long long) { *x = reinterpret_cast<cudaGraphExec_t>(std::malloc(1)); return cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t g) { std::free(g); return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t x) { std::free(x); return cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { g_log += "g "; return cudaSuccess; }
cudaError_t cudaThreadExchangeStreamCaptureMode(cudaStreamCaptureMode *m)
{
    const cudaStreamCaptureMode old = g_relaxed ? cudaStreamCaptureModeRelaxed : cudaStreamCaptureModeGlobal;
    g_relaxed = *m == cudaStreamCaptureModeRelaxed;
    *m = old;
    return cudaSuccess;
}
cudaError_t cudaGetDriverEntryPointByVersion(const char *, void **p, unsigned, unsigned long long, cudaDriverEntryPointQueryResult *q)
{
    *p = reinterpret_cast<void *>(&fake_encode);
    if (q) *q = cudaDriverEntryPointSuccess;
    return cudaSuccess;
}
}

static cudaError_t say(const std::string &what)
{
    if (!g_capture) g_log += what + " ";
    return cudaSuccess;
}
static cudaError_t resident(const char *what, int n)
{
    if (hit(fake_fail_resident)) return cudaErrorCooperativeLaunchTooLarge;
    return say(what + std::to_string(n));
}
namespace lbm13 {
int device_sm_count() { return 152; }
int linear_growth(const lbm13_params &, const double *, double, double, int, double *g) { *g = 0.0; return LBM13_OK; }
int linear_growth_batch(const lbm13_params *, const double *, const double *, const double *, int, int, double *, cudaStream_t) { return LBM13_OK; }
bool batch_shape_supported(int, int) { return true; }
int reduce_blocks(int nx, int ny) { return nx * ny / 256 + 1; }
template <typename T, typename C> int multi_grid(int, int, bool) { return 152; }
template int multi_grid<float, float>(int, int, bool);
template int multi_grid<double, double>(int, int, bool);
template <typename T, typename C>
cudaError_t launch_multi(const StepArgs<T, C> &, const StepArgs<T, C> &, bool, int n, int, const GridSync &, cudaStream_t) { return say("M" + std::to_string(n)); }
cudaError_t launch_pair_step(const StepArgs<float, float> &, const CUtensorMap &, bool, unsigned *, cudaStream_t, int, unsigned long long) { return say("2"); }
cudaError_t launch_batch_tma(const BatchDesc<float, float> *, const LatticeMaps *, const int2 *, int, int, int, unsigned *, cudaStream_t, int, unsigned long long) { return say("b"); }
cudaError_t launch_batch_ring(const BatchDesc<float, float> *, const LatticeMaps *, const int2 *, int, int, int, int, unsigned *, cudaStream_t, int, unsigned long long) { return say("b"); }
cudaError_t launch_barrier_check(int, unsigned, int, const GridSync &, cudaStream_t) { return cudaSuccess; }
template <typename T, typename C> cudaError_t launch_step(const StepArgs<T, C> &, bool, cudaStream_t) { return say("s"); }
template <typename T, typename C>
cudaError_t launch_batch(const BatchDesc<T, C> *, const int2 *, int, int, int, int, int, int, cudaStream_t) { return say("b"); }
template <typename T> cudaError_t launch_halo(T *, int, int, long long, long long, int, bool, T *, cudaStream_t) { return cudaSuccess; }
template <typename T>
cudaError_t launch_init(T *, int, int, long long, long long, const InitFix &, const double *, const double *, const double *, const double *, cudaStream_t) { return cudaSuccess; }
template <typename T> cudaError_t launch_moments(const ReadArgs<T> &, double *, unsigned, cudaStream_t) { return cudaSuccess; }
// the block counts have to be zero when a pass starts
template <typename T> cudaError_t launch_reduce(const ReduceJob<T> &j, cudaStream_t)
{
    std::memset(j.out, 0, 16 * sizeof(double));
    if (j.err) j.out[16] = 0.0;
    return say(*j.b.done == 0 ? "reduce" : "REDUCE-NOT-CLEARED");
}
template <typename T> cudaError_t launch_reduce_batch(const ReduceJob<T> *jobs, int count, int, cudaStream_t)
{
    for (int i = 0; i < count; ++i) {
        std::memset(jobs[i].out, 0, 16 * sizeof(double));
        if (jobs[i].err) jobs[i].out[16] = 0.0;
    }
    return say("reduce-all");
}
template <typename T>
cudaError_t launch_project(const ReadArgs<T> &, int, int, double *, int, unsigned *done, double *, cudaStream_t)
{
    return say(*done == 0 ? "project" : "PROJECT-NOT-CLEARED");
}
template <typename T, typename C>
cudaError_t launch_resident(const StepArgs<T, C> &a, bool, int n, const ResShape &, void *xchg, unsigned, unsigned *err,
                            unsigned long long, cudaStream_t, int)
{
    const unsigned *w = static_cast<const unsigned *>(xchg);
    for (size_t i = 3; i < res_exchange_bytes(a.nx, a.ny, sizeof(T)) / 4; i += 4)
        if (w[i] == 0xa5a5a5a5u) return say("RESIDENT-NOT-CLEARED");
    if (*err) return say("ERROR-WORD-NOT-CLEARED");
    return resident("R", n);
}
cudaError_t launch_resident_plan(const BatchDesc<float, float> *, const ResPlanTile *, int, int, int, size_t, bool, int, int n,
                                 void *, unsigned, unsigned *, unsigned long long, cudaStream_t) { return resident("P", n); }
template <typename T, typename C>
int resident_capacity(const ResShape &, bool, const WallArgs<C> *) { return 152 * fake_blocks_per_sm; }
int resident_plan_capacity(int, int, size_t, bool) { return 152 * fake_blocks_per_sm; }
#define BOTH(T) \
    template int resident_capacity<T, T>(const ResShape &, bool, const WallArgs<T> *); \
    template cudaError_t launch_multi<T, T>(const StepArgs<T, T> &, const StepArgs<T, T> &, bool, int, int, const GridSync &, cudaStream_t); \
    template cudaError_t launch_step<T, T>(const StepArgs<T, T> &, bool, cudaStream_t); \
    template cudaError_t launch_batch<T, T>(const BatchDesc<T, T> *, const int2 *, int, int, int, int, int, int, cudaStream_t); \
    template cudaError_t launch_halo<T>(T *, int, int, long long, long long, int, bool, T *, cudaStream_t); \
    template cudaError_t launch_init<T>(T *, int, int, long long, long long, const InitFix &, const double *, const double *, const double *, const double *, cudaStream_t); \
    template cudaError_t launch_moments<T>(const ReadArgs<T> &, double *, unsigned, cudaStream_t); \
    template cudaError_t launch_reduce<T>(const ReduceJob<T> &, cudaStream_t); \
    template cudaError_t launch_reduce_batch<T>(const ReduceJob<T> *, int, int, cudaStream_t); \
    template cudaError_t launch_project<T>(const ReadArgs<T> &, int, int, double *, int, unsigned *, double *, cudaStream_t); \
    template cudaError_t launch_resident<T, T>(const StepArgs<T, T> &, bool, int, const ResShape &, void *, unsigned, unsigned *, unsigned long long, cudaStream_t, int);
BOTH(float)
BOTH(double)
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    if shutil.which("g++") is None or not os.path.exists(os.path.join(CUDA_INC, "cuda_runtime.h")):
        pytest.skip("needs g++ and the CUDA headers")
    d = tmp_path_factory.mktemp("dispatch")
    (d / "fake.cpp").write_text(FAKE)
    opts = ["g++", "-O1", "-std=c++17", "-fPIC", "-w", "-D__noinline__=", "-I", CSRC, "-I", CUDA_INC]
    subprocess.check_call([*opts, "-x", "c++", "-c", os.path.join(CSRC, "lbm13_api.cu"), "-o", str(d / "api.o")])
    subprocess.check_call([*opts, "-c", str(d / "fake.cpp"), "-o", str(d / "fake.o")])
    # -Bsymbolic: the stand-in's calls, whatever CUDA library the process has loaded
    subprocess.check_call(["g++", "-shared", "-Wl,-Bsymbolic", str(d / "api.o"), str(d / "fake.o"), "-ldl", "-o", str(d / "dispatch.so")])
    L = C.CDLL(str(d / "dispatch.so"))
    L.fake_log.restype = C.c_char_p
    L.lbm13_last_error.restype = C.c_char_p
    L.lbm13_plan_last_error.restype = C.c_char_p
    L.lbm13_time.restype = C.c_int64
    return L


class Lat:
    """A lattice of the stand-in (cudaMalloc, stream NULL)."""

    def __init__(self, L, nx, ny, precision=FP32, bnd=None, mode=AUTO):
        p = pstar(0.05, 0.71)
        self.L, self.n = L, nx * ny
        self.h = C.c_void_p()
        st = L.lbm13_create(nx, ny, C.byref(B.make_params(p)), C.byref(B.make_boundary(bnd or W.boundary())), precision,
                            None, None, C.byref(self.h))
        assert st == 0
        assert L.lbm13_set_persistent(self.h, mode) == 0
        L.fake_clear()

    def step(self, n):
        """(status, launches) of a run of n steps."""
        self.L.fake_clear()
        st = self.L.lbm13_step(self.h, C.c_int64(n))
        return st, self.log()

    def log(self):
        return self.L.fake_log().decode().split()

    def close(self):
        self.L.lbm13_destroy(self.h)


def _set(L, **kw):
    for k, v in kw.items():
        C.c_int.in_dll(L, "fake_" + k).value = v


@pytest.fixture(autouse=True)
def _defaults(lib):
    yield
    _set(lib, fail_memset=0, fail_malloc=0, fail_resident=0, cooperative=1, capturing=0, blocks_per_sm=1, other_capture=0)


def _cavity(**kw):
    return W.cavity(rest_temperature(pstar(0.05, 0.71)), 0.01, 1e-4, **kw)


def test_no_memory_is_kept_when_the_stand_in_frees_all(lib):
    a = Lat(lib, 64, 64)
    assert a.step(64)[0] == 0
    out = (C.c_double * 24)()
    assert lib.lbm13_residual(a.h, out) == 0 and lib.lbm13_project(a.h, 0, 1, out) == 0
    assert "reduce" in a.log() and "project" in a.log()
    a.close()
    assert lib.fake_allocations() == 0


@pytest.mark.parametrize("which", [1, 2])
def test_a_buffer_that_could_not_be_cleared_is_not_stepped_with(lib, which):
    """The first clear of a long run is that of the error word, the second that of the
    exchange buffer."""
    a = Lat(lib, 64, 64)
    _set(lib, fail_memset=which)
    for _ in range(2):
        st, log = a.step(64)
        assert st == 0 and not any("NOT-CLEARED" in x for x in log), log
    a.close()
    assert lib.fake_allocations() == 0


@pytest.mark.parametrize("call", ["residual", "project"])
def test_a_work_space_that_could_not_be_cleared_is_made_again(lib, call):
    a = Lat(lib, 64, 64)
    out = (C.c_double * 24)()
    f = (lambda: lib.lbm13_residual(a.h, out)) if call == "residual" else (lambda: lib.lbm13_project(a.h, 0, 1, out))
    _set(lib, fail_memset=1)
    assert f() == 6  # LBM13_ECUDA
    assert f() == 0
    assert not any("NOT-CLEARED" in x for x in a.log()), a.log()
    a.close()
    assert lib.fake_allocations() == 0


def test_launches_of_a_run(lib):
    """By mode, length and size; asking for their number makes and allocates nothing."""
    n = C.c_int64()
    for nx, ny, prec, mode, steps, want in [
            (64, 64, FP32, AUTO, 64, ["R64"]), (64, 64, FP32, AUTO, 31, ["s"] * 31), (64, 64, FP32, OFF, 64, ["g", "g"]),
            (64, 64, FP32, ON, 2, ["R2"]), (900, 900, FP32, AUTO, 64, ["g", "g"]), (900, 900, FP32, ON, 64, ["M64"]),
            (64, 64, FP64, AUTO, 32, ["R32"]), (64, 64, FP64, ON, 1, ["s"])]:
        a = Lat(lib, nx, ny, prec, _cavity(), mode)
        held = lib.fake_allocations()
        assert lib.lbm13_step_launches(a.h, C.c_int64(steps), C.byref(n)) == 0
        assert lib.fake_allocations() == held and a.log() == []
        st, log = a.step(steps)
        assert st == 0 and log == want, (nx, prec, mode, steps, log)
        per_graph = {"g": 32}
        assert n.value == sum(per_graph.get(x, 1) for x in log)
        a.close()


def test_large_fp64_lattices_step_launch_by_launch(lib):
    """Where shared memory holds them but single launches are faster."""
    M, BB = W.WALL_MIXED, W.WALL_BB
    T0 = rest_temperature(pstar(0.05, 0.71))
    box = W.boundary(west=W.wall(M, 0.0, T0), east=W.wall(BB), south=W.wall(M, 0.01, T0), north=W.wall(BB))
    for nx, ny, prec, bnd, mode, want in [
            (362, 362, FP64, _cavity(), AUTO, "R"), (363, 362, FP64, _cavity(), AUTO, "g"), (500, 500, FP64, None, AUTO, "g"),
            (1024, 128, FP64, None, AUTO, "R"), (440, 440, FP64, box, AUTO, "R"), (440, 440, FP64, _cavity(), ON, "R"),
            (600, 600, FP32, _cavity(), AUTO, "R")]:
        a = Lat(lib, nx, ny, prec, bnd, mode)
        st, log = a.step(64)
        assert st == 0 and log[0][0] == want, (nx, ny, prec, mode, log)
        a.close()


@pytest.mark.parametrize("mode", [AUTO, ON])
def test_a_refused_launch_from_shared_memory_leaves_the_steps_to_others(lib, mode):
    a = Lat(lib, 64, 64, FP32, _cavity(), mode)
    _set(lib, fail_resident=1)
    st, log = a.step(70)
    assert st == 0 and log == (["M70"] if mode == ON else ["g", "g"] + ["s"] * 6), log
    assert lib.lbm13_time(a.h) == 70
    a.close()
    b = Lat(lib, 64, 64, FP32, _cavity(), mode)
    _set(lib, fail_resident=2)  # the second of three launches
    st, log = b.step(1024 + 1024 + 64)
    assert st == 0 and log[0] == "R1024" and not any(x.startswith("R") for x in log[1:])
    assert lib.lbm13_time(b.h) == 2112
    b.close()


def test_no_launch_from_shared_memory_where_its_blocks_do_not_fit_at_once(lib):
    _set(lib, blocks_per_sm=0)
    a = Lat(lib, 64, 64, FP32, _cavity())
    assert a.step(64) == (0, ["g", "g"])
    a.close()


def test_a_run_allocates_beside_a_capture_elsewhere(lib):
    a = Lat(lib, 64, 64, FP32, _cavity())
    _set(lib, other_capture=1)
    assert a.step(64) == (0, ["R64"])
    _set(lib, other_capture=0, capturing=1)  # its own stream is captured: the launches that are recorded
    assert a.step(33) == (0, ["g", "s"])
    a.close()


def _plan(lib, lats):
    arr = (C.c_void_p * len(lats))(*[a.h for a in lats])
    p = C.c_void_p()
    assert lib.lbm13_plan_create(arr, len(lats), None, None, C.byref(p)) == 0
    return p


def test_a_refused_plan_launch_leaves_the_steps_to_others(lib):
    lats = [Lat(lib, 64, 64, FP32, _cavity()) for _ in range(3)]
    p = _plan(lib, lats)
    lib.fake_clear()
    assert lib.lbm13_plan_step(p, C.c_int64(64)) == 0 and lats[0].log() == ["P64"]
    _set(lib, fail_resident=1)
    lib.fake_clear()
    assert lib.lbm13_plan_step(p, C.c_int64(65)) == 0 and lats[0].log() == ["g", "g", "b"]
    assert [lib.lbm13_time(a.h) for a in lats] == [129] * 3
    lib.lbm13_plan_destroy(p)
    for a in lats:
        a.close()
    assert lib.fake_allocations() == 0
