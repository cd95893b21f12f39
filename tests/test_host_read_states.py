"""Read-outs and initial states (csrc/lbm13_read.cuh, csrc/lbm13_fixed_io.cuh) on the
host, at the states that flows hold: a small velocity beside large deviations of
density and temperature, and the other way round.  Against 113-bit arithmetic no
reading and no momentum is less exact than FP64 arithmetic with one rounding per
operation gives it."""
import ctypes as C
import os
import shutil
import subprocess

import numpy as np
import pytest

import test_host_fixed_states as S
from paper_1401_0188_gb300 import lbm13, pstar
from paper_1401_0188_gb300 import params as P
from paper_1401_0188_gb300 import workloads as W

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1401_0188_gb300", "csrc")
CUDA_INC = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")
Q = 13

SRC = r"""
#include <algorithm>
#include <cmath>
#include <cstring>
#include <cuda_runtime.h>
#include "lbm13_coef.h"
using std::isfinite;
#include "lbm13_read.cuh"
using namespace lbm13;
#if __LDBL_MANT_DIG__ >= 113
typedef long double quad;
#else
typedef __float128 quad;
#endif

// f [13][n]; out [n][8]: rho - 1, E - E0, j_x, j_y, u_x, u_y, T - T0, p - T0: the
// kernels' node_dev (ei) and FP64 operation by operation (ep), errors
template <typename T>
static void read_all(const lbm13_params &p, const lbm13_boundary &b, int n, const T *f, double *value, double *ei, double *ep)
{
    ReadArgs<T> a{};
    a.f = f;
    a.nx = n;
    a.ny = 1;
    a.pitch = a.plane = n;
    a.rest.E0 = p.E0;
    a.rest.T0 = (p.E0 + 28.0) / 26.0;
    a.gx = b.gx;
    a.gy = b.gy;
    a.rho_ref = b.rho_ref;
    a.heat = b.heat;
    a.force = b.gx != 0.0 || b.gy != 0.0;
    read_fix(p.E0, b, a.fx);
    for (int i = 0; i < n; ++i) {
        double g[Q];
        quad e[Q];
        for (int j = 0; j < Q; ++j) g[j] = f[size_t(j) * n + i], e[j] = g[j];
        Mom<quad> m;
        forward(e, m);
        const quad rho = 1 + m.rho, w = (rho - quad(b.rho_ref)) / 2, T0 = (quad(p.E0) + 28) / 26;
        const quad pd = (m.E + 28 * m.rho) / 26 - (m.jx * m.jx + m.jy * m.jy) / (2 * rho) - quad(b.heat) / 2;
        const quad x[8] = {m.rho, m.E, m.jx, m.jy, (m.jx - w * quad(b.gx)) / rho, (m.jy - w * quad(b.gy)) / rho,
                           (pd - T0 * m.rho) / rho, pd};
        Mom<double> d;
        forward(g, d);
        const double r = 1.0 + d.rho, h = 0.5 * (r - b.rho_ref), t0 = (p.E0 + 28) / 26;
        const double dp = (d.E + 28.0 * d.rho) / 26.0 - (d.jx * d.jx + d.jy * d.jy) / (2.0 * r) - 0.5 * b.heat;
        const double y[8] = {d.rho, d.E, d.jx, d.jy, (d.jx - h * b.gx) / r, (d.jy - h * b.gy) / r, (dp - t0 * d.rho) / r, dp};
        const NodeDev o = node_dev(a, i);
        const double z[8] = {o.rho, o.E, o.jx, o.jy, o.ux, o.uy, o.T, o.p};
        for (int c = 0; c < 8; ++c) {
            value[i * 8 + c] = z[c];
            ei[i * 8 + c] = double(quad(z[c]) - x[c]);
            ep[i * 8 + c] = double(quad(y[c]) - x[c]);
        }
    }
}
extern "C" void read64(const lbm13_params *p, const lbm13_boundary *b, int n, const double *f, double *v, double *ei, double *ep)
{
    read_all(*p, *b, n, f, v, ei, ep);
}
extern "C" void read32(const lbm13_params *p, const lbm13_boundary *b, int n, const float *f, double *v, double *ei, double *ep)
{
    read_all(*p, *b, n, f, v, ei, ep);
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    if shutil.which("g++") is None or not os.path.exists(os.path.join(CUDA_INC, "cuda_runtime.h")):
        pytest.skip("needs g++ and the CUDA headers")
    d = tmp_path_factory.mktemp("read_states")
    src, so = d / "read.cpp", d / "read.so"
    src.write_text(SRC)
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-D__noinline__=", "-fPIC", "-shared", "-w", "-I", CSRC, "-I",
                           CUDA_INC, str(src), "-o", str(so)])
    return C.CDLL(str(so))


BOUNDS = {"plain": W.boundary(), "buoyancy": W.boundary(gy=-3e-5, rho_ref=1.0), "source": W.boundary(gx=2e-6, gy=1e-6, heat=1e-7)}
PARAMS = {"pstar": lambda: pstar(0.05, 0.71), "high_pr": lambda: P.select(0.3, 1.0)}
ptr = lambda a: a.ctypes.data_as(C.c_void_p)  # noqa: E731
rms = lambda e: np.sqrt(np.mean(e ** 2, axis=0))  # noqa: E731


def _read(lib, p, b, f, single):
    """f [n][13] in the storage type: (values, errors, errors of plain FP64), [n][8]."""
    g = np.ascontiguousarray(f.T.astype(np.float32 if single else np.float64))
    out = [np.zeros((len(f), 8)) for _ in range(3)]
    Pp, Bb = lbm13.make_params(p), lbm13.make_boundary(b)
    (lib.read32 if single else lib.read64)(C.byref(Pp), C.byref(Bb), len(f), ptr(g), *[ptr(o) for o in out])
    return out


def _check_reading(lib, params, sizes, bound, single):
    p = PARAMS[params]()
    f = S._states(p, S.SIZES[sizes], 4000, np.random.default_rng(3), 1e-3)
    v, ei, ep = _read(lib, p, BOUNDS[bound], f, single)
    # 4000 nodes estimate each rms to 1.1%; a reading's own last rounding is in both
    assert (rms(ei) <= 1.05 * rms(ep)).all(), rms(ei) / rms(ep)


@pytest.mark.parametrize("bound", list(BOUNDS))
@pytest.mark.parametrize("sizes", list(S.SIZES))
@pytest.mark.parametrize("params", list(PARAMS))
def test_fp64_readings_are_no_less_exact_than_fp64_arithmetic(lib, params, sizes, bound):
    _check_reading(lib, params, sizes, bound, False)


def test_fp64_readings_far_from_rest_and_of_bad_nodes(lib):
    p = pstar(0.05, 0.71)
    f = 1e-3 * np.random.default_rng(1).standard_normal((6, Q))
    f[0] = 0.0
    f[1, 3] = np.nan
    f[2, 5] = -np.inf
    f[3, 0] = 1.5           # density 2.5: the quotients divide
    f[4, 0] = -0.8
    f[5] *= 1e-200
    v, ei, ep = _read(lib, p, W.boundary(), f, False)
    assert (v[0] == 0).all() and np.isnan(v[1]).any() and not np.isfinite(v[2]).all()
    u = np.ix_([3, 4, 5], [4, 5])  # the velocities (T and p are differences of larger terms)
    assert (np.abs(ei[u]) <= 2 * np.abs(ep[u]) + 2.0 ** -52 * np.abs(v[u])).all()


INIT_SRC = r"""
// in [n][4]: rho, ux, uy, T; errors [n][17] of the 13 deviations, j_x, j_y, E and f1 - f3
extern "C" void init64(const lbm13_params *p, const double *D, const lbm13_boundary *b, int n, const double *in, double *ei,
                       double *ep)
{
    Coef<double> kd;
    collision_coef(*p, D, *b, kd);
    InitFix k;
    init_fix(*p, D, k);
    for (int i = 0; i < n; ++i) {
        const double r = in[4 * i], u = in[4 * i + 1], v = in[4 * i + 2], t = in[4 * i + 3];
        const quad R = quad(r) - 1, jx = quad(r) * u, jy = quad(r) * v;
        const quad dE = quad(r) * (26 * quad(t) - 28) - quad(p->E0) + 13 * quad(r) * (quad(u) * u + quad(v) * v);
        const quad Qe = quad(p->c1) + quad(D[2]) * (1 + R) + quad(D[3]) * (quad(p->E0) + dE);
        const quad Re = quad(D[5]) + quad(D[4]) * (1 + R) + quad(p->k2) * (quad(p->E0) + dE);
        Mom<quad> d;
        d.rho = R / 13;
        d.E = dE / 4004;
        d.eps = (quad(D[6]) * R + quad(p->c_epsE) * dE) / 42196;
        d.vpi = (quad(p->c_vpi_rho) * R + quad(p->c_vpi_E) * dE) / 548;
        d.jx = jx / 14;
        d.jy = jy / 14;
        d.qx = jx * Qe / 20;
        d.qy = jy * Qe / 20;
        d.rx = jx * Re / 70;
        d.ry = jy * Re / 70;
        d.XX = (jx * jx - jy * jy) / quad(r) / 68;
        d.XY = jx * jy / quad(r) / 4;
        d.XXe = 0;
        quad e[Q] = {};
        inverse_add<true>(d, e);
        double g[2][Q];
        init_node(r, u, v, t, k, g[0]);
        equilibrium_dev(r - 1.0, r * (26.0 * t - 28.0) - p->E0 + 13.0 * r * (u * u + v * v), r * u, r * v, kd, g[1]);
        for (int w = 0; w < 2; ++w) {
            double *o = (w ? ep : ei) + i * 17;
            quad q[Q];
            Mom<quad> m;
            for (int j = 0; j < Q; ++j) q[j] = g[w][j], o[j] = double(q[j] - e[j]);
            forward(q, m);
            o[13] = double(m.jx - jx);
            o[14] = double(m.jy - jy);
            o[15] = double(m.E - dE);
            o[16] = double((q[1] - q[3]) - (e[1] - e[3]));
        }
    }
}
"""


@pytest.mark.parametrize("sizes", list(S.SIZES))
@pytest.mark.parametrize("params", list(PARAMS))
def test_fp64_initial_states_are_no_less_exact_than_fp64_arithmetic(tmp_path, params, sizes):
    if shutil.which("g++") is None or not os.path.exists(os.path.join(CUDA_INC, "cuda_runtime.h")):
        pytest.skip("needs g++ and the CUDA headers")
    src, so = tmp_path / "init.cpp", tmp_path / "init.so"
    src.write_text(SRC + INIT_SRC)
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-D__noinline__=", "-fPIC", "-shared", "-w", "-I",
                           CSRC, "-I", CUDA_INC, str(src), "-o", str(so)])
    p = PARAMS[params]()
    st, D = lbm13.lbm13_derive(p)
    n, a = 4000, S.SIZES[sizes]
    x = np.array([1.0, 0.0, 0.0, P.rest_temperature(p)]) + np.array([a[0], a[1], a[1], a[2]]) * np.random.default_rng(5).standard_normal((n, 4))
    x = np.ascontiguousarray(x)
    ei, ep = np.zeros((n, 17)), np.zeros((n, 17))
    Pp, Bb = lbm13.make_params(p), lbm13.make_boundary(W.boundary())
    C.CDLL(str(so)).init64(C.byref(Pp), ptr(np.ascontiguousarray(D)), C.byref(Bb), n, ptr(x), ptr(ei), ptr(ep))
    assert (rms(ei) <= 1.05 * rms(ep)).all(), rms(ei) / rms(ep)


@pytest.mark.parametrize("bound", list(BOUNDS))
@pytest.mark.parametrize("sizes", list(S.SIZES))
@pytest.mark.parametrize("params", list(PARAMS))
def test_fp32_readings_are_no_less_exact_than_fp64_arithmetic(lib, params, sizes, bound):
    _check_reading(lib, params, sizes, bound, True)


@pytest.mark.parametrize("single", [False, True])
@pytest.mark.parametrize("sizes", [(2e-3, 1e-2, 2e-3), (1e-2, 3e-2, 1e-2), (1e-4, 1e-3, 2e-3), (1e-2, 1e-7, 1e-3), (1e-3, 2e-2, 1e-5)])
def test_no_reading_leaves_its_range(lib, sizes, single):
    """A sum beyond 63 bits would be off by a large part of the node's populations: 400,000
    nodes, the squares of the velocity above the second moment among them."""
    p = pstar(0.05, 0.71)
    f = S._states(p, sizes, 400_000, np.random.default_rng(100), 1e-2)
    v, ei, ep = _read(lib, p, BOUNDS["buoyancy"], f, single)
    assert (np.abs(ei).max(axis=1) <= 2.0 ** -40 * np.abs(f).max(axis=1)).all()


def test_fp32_readings_of_floats_below_the_normal_range(lib):
    """Nodes of 1e-30 and less, some of whose populations are subnormal."""
    p = pstar(0.05, 0.71)
    rng = np.random.default_rng(8)
    f = rng.standard_normal((2000, Q)) * 10.0 ** rng.integers(-36, -18, (2000, 1)).astype(float)
    f[:, 3:9] *= 1e-7
    v, ei, ep = _read(lib, p, W.boundary(), f, True)
    scale = np.abs(f).max(axis=1)[:, None]
    assert (rms(ei / scale) <= 1.05 * rms(ep / scale)).all()


@pytest.mark.parametrize("mirror", list(S.MIRRORS))
@pytest.mark.parametrize("bound", list(BOUNDS))
@pytest.mark.parametrize("single", [False, True])
def test_mirrored_nodes_read_to_mirrored_values(lib, single, bound, mirror):
    p, b, m = pstar(0.05, 0.71), BOUNDS[bound], S.MIRRORS[mirror]
    image = dict(b, gx=b["gx"] * (-1 if "x" in mirror else 1), gy=b["gy"] * (-1 if "y" in mirror else 1))
    f = np.concatenate([S._states(p, a, 2000, np.random.default_rng(9), 1e-3) for a in S.SIZES.values()])
    sign = np.ones(8)
    sign[[2, 4]] *= -1 if "x" in mirror else 1
    sign[[3, 5]] *= -1 if "y" in mirror else 1
    assert np.array_equal(_read(lib, p, b, f, single)[0] * sign, _read(lib, p, image, f[:, m], single)[0])


MIRROR_SRC = r"""
template <typename T>
static void init_all(const lbm13_params &p, const double *D, int n, const double *in, T *out)
{
    InitFix k;
    init_fix(p, D, k);
    for (int i = 0; i < n; ++i) {
        T g[Q];
        init_node(in[4 * i], in[4 * i + 1], in[4 * i + 2], in[4 * i + 3], k, g);
        for (int j = 0; j < Q; ++j) out[i * Q + j] = g[j];
    }
}
extern "C" void set64(const lbm13_params *p, const double *D, int n, const double *in, double *out) { init_all(*p, D, n, in, out); }
extern "C" void set32(const lbm13_params *p, const double *D, int n, const double *in, float *out) { init_all(*p, D, n, in, out); }
"""


@pytest.mark.parametrize("single", [False, True])
def test_mirrored_initial_states_are_mirror_images(tmp_path, single):
    if shutil.which("g++") is None or not os.path.exists(os.path.join(CUDA_INC, "cuda_runtime.h")):
        pytest.skip("needs g++ and the CUDA headers")
    src, so = tmp_path / "set.cpp", tmp_path / "set.so"
    src.write_text(SRC + MIRROR_SRC)
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-D__noinline__=", "-fPIC", "-shared", "-w", "-I",
                           CSRC, "-I", CUDA_INC, str(src), "-o", str(so)])
    L, p = C.CDLL(str(so)), pstar(0.05, 0.71)
    st, D = lbm13.lbm13_derive(p)
    n, dtype = 20000, np.float32 if single else np.float64
    rng = np.random.default_rng(6)
    x = np.array([1.0, 0.0, 0.0, P.rest_temperature(p)]) + 10.0 ** rng.integers(-5, -1, (n, 1)).astype(float) * rng.standard_normal((n, 4))
    x[::2, 1:3] = np.round(x[::2, 1:3] * 2.0 ** 12) * 2.0 ** -12  # few significant bits
    Pp = lbm13.make_params(p)

    def state(y):
        out = np.zeros((n, Q), dtype=dtype)
        (L.set32 if single else L.set64)(C.byref(Pp), ptr(np.ascontiguousarray(D)), n, ptr(np.ascontiguousarray(y)), ptr(out))
        return out

    f = state(x)
    for mirror, m in S.MIRRORS.items():
        sign = np.array([1.0, -1.0 if "x" in mirror else 1.0, -1.0 if "y" in mirror else 1.0, 1.0])
        assert np.array_equal(f[:, m], state(x * sign))
