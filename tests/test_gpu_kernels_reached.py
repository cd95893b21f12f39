"""Kernels that the default modes reach at some sizes only, each on lattices that do
reach it: grid-barrier launches of lattices that shared memory does not hold, the
ring-staged strips through 32-step graphs, the walled per-step kernels and the shared
rows in the bounds-checked build, and the bounded wait of stepping from shared memory
made to run out."""
import json
import os
import subprocess
import sys

import numpy as np
import pytest

from paper_1401_0188_gb300 import pstar as product_pstar
from paper_1401_0188_gb300 import workloads as W

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def L():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1401_0188_gb300 import build, lbm13
    build.build()
    lbm13.lib()
    return lbm13


def _lattice(L, nx, ny, kind, precision, mode, stream=None):
    p = product_pstar(0.05, 0.71)
    T0 = (p["E0"] + 28) / 26
    M, B = W.WALL_MIXED, W.WALL_BB
    bnd = {"periodic": W.boundary(gx=2e-5, gy=-1e-5, heat=2e-6), "cavity": W.cavity(T0, 0.01, 1e-4),
           "cavity_zero_flux": W.cavity(T0, 0.01, 1e-4, wall_density=1), "couette": W.couette(T0, 0.02, 0.01),
           "box": W.boundary(west=W.wall(M, -0.01, T0 + 0.005), east=W.wall(B, 0.015), south=W.wall(M, 0.02, T0),
                             north=W.wall(B), gx=1e-5, gy=-2e-5, rho_ref=1.0)}[kind]
    g = L.Lattice(nx, ny, p, bnd, precision=precision, stream=stream)
    g.set_persistent(mode)
    g.set_state(*W.random_fields(nx, ny, T0, seed=nx + ny, du=0.01, drho=0.005, dT=0.003))
    return g


@pytest.mark.parametrize("kind", ["periodic", "cavity", "cavity_zero_flux", "couette", "box"])
@pytest.mark.parametrize("precision", [0, 1])
def test_grid_barrier_launches_of_lattices_that_shared_memory_does_not_hold(L, kind, precision):
    nx, ny = (901, 803) if precision else (571, 502)  # more populations than the SMs hold
    a = _lattice(L, nx, ny, kind, precision, L.PERSISTENT_ON)
    b = _lattice(L, nx, ny, kind, precision, L.PERSISTENT_OFF)
    held = a.info()["device_bytes"]
    assert a.step_launches(40) == 1
    for n in (2, 33, 1031 if kind == "cavity" else 7):  # the longest takes two launches
        a.step(n)
        b.step(n)
        assert a.save() == b.save(), n
    # the grid of the barrier kernel, and no exchange buffer: nothing was stepped from
    # shared memory
    assert a.info()["persistent_grid"] > 0 and a.info()["device_bytes"] - held < 4096
    a.close()
    b.close()


@pytest.mark.parametrize("BY", [8, 4])
def test_ring_strips_through_graphs_on_lattices_that_step_launch_by_launch(L, BY):
    sizes = [(300, 260, "cavity"), (257, 131, "periodic"), (128, 640, "couette"), (64, 64, "box")]
    a = [_lattice(L, nx, ny, k, 1, L.PERSISTENT_OFF) for nx, ny, k in sizes]
    b = [_lattice(L, nx, ny, k, 1, L.PERSISTENT_OFF) for nx, ny, k in sizes]
    plan = L.Plan(a)
    for groups in (3, 16):
        plan.set_config(0, BY, 0, 2, groups)
        plan.step(35)  # one 32-step graph and three launches
        for x, y in zip(a, b):
            y.step(35)
            assert x.save() == y.save()
    with pytest.raises(L.Lbm13Error):
        plan.resident_check(0.02)  # the plan does not step from shared memory
    plan.close()


@pytest.mark.parametrize("kind", ["periodic", "cavity", "box"])
@pytest.mark.parametrize("precision", [0, 1])
def test_the_wait_between_tiles_is_bounded(L, precision, kind):
    """Without its last tile a launch's waits run out: the error is reported once, the
    state is kept, and later runs equal single launches (the exchange goes on with
    numbers that the aborted launch did not use)."""
    a = _lattice(L, 150, 130, kind, precision, L.PERSISTENT_AUTO)
    b = _lattice(L, 150, 130, kind, precision, L.PERSISTENT_OFF)
    a.step(64)
    b.step(64)
    image = a.save()
    assert image == b.save()
    assert a.resident_check(0.5, withhold=0) is False
    assert a.resident_check(0.005, withhold=1) is True
    assert a.save() == image
    assert a.resident_check(0.005, withhold=2) is True
    with pytest.raises(L.Lbm13Error) as e:
        a.residual()
    assert e.value.status == 5  # LBM13_ETIMEOUT
    a.residual()
    assert a.save() == image
    for n in (200, 33):
        a.step(n)
        b.step(n)
        assert a.save() == b.save()
    with pytest.raises(L.Lbm13Error):
        b.resident_check(0.005)
    a.close()
    b.close()


def test_the_wait_between_tiles_of_a_plan_is_bounded(L):
    sizes = [(64, 64, "cavity"), (97, 60, "periodic"), (120, 90, "box")]
    a = [_lattice(L, nx, ny, k, 1, L.PERSISTENT_AUTO) for nx, ny, k in sizes]
    b = [_lattice(L, nx, ny, k, 1, L.PERSISTENT_OFF) for nx, ny, k in sizes]
    plan = L.Plan(a)
    plan.step(64)
    for g in b:
        g.step(64)
    assert plan.resident_check(0.5, withhold=0) is False
    assert plan.resident_check(0.005, withhold=1) is True
    assert plan.resident_check(0.005, withhold=2) is True
    with pytest.raises(L.Lbm13Error) as e:
        plan.residual()
    assert e.value.status == 5
    r = plan.residual()
    assert np.isfinite(r).all()
    plan.step(200)
    for x, y in zip(a, b):
        y.step(200)
        assert x.save() == y.save()
    plan.close()


SCRIPT = r"""
import json
import torch
from paper_1401_0188_gb300 import lbm13, params as P, workloads as W

p = P.pstar(0.05, 0.71)
T0 = P.rest_temperature(p)
M, B = W.WALL_MIXED, W.WALL_BB
box = W.boundary(west=W.wall(M, -0.01, T0 + 0.005), east=W.wall(M, 0.015, T0 - 0.005), south=W.wall(M, 0.02, T0),
                 north=W.wall(M, -0.01, T0))
cases = [(48, 40, W.cavity(T0, 0.01, 2e-4)), (37, 30, W.couette(T0, 0.05, 0.01)), (34, 29, box), (4, 4, box),
         (100, 70, W.cavity(T0, 0.01, 1e-4, wall_density=1)), (40, 24, W.heated_slab(T0, 1e-5, 0.02)), (131, 97, W.boundary(gx=1e-5))]
launches, lats = {"step": 0, "resident": 0, "barrier": 0}, []


def run(nx, ny, bnd, prec, mode, n, kind):
    g = lbm13.Lattice(nx, ny, p, bnd, precision=prec)
    g.set_persistent(mode)
    g.set_state(*W.random_fields(nx, ny, T0, 7, du=0.01, drho=0.005, dT=0.003))
    launches[kind] += g.step_launches(n) == (n if kind == "step" else 1)
    g.step(n)
    g.step(3)
    lats.append(g)


for prec in (lbm13.FP64, lbm13.FP32_DEVIATION):
    for nx, ny, bnd in cases:
        run(nx, ny, bnd, prec, lbm13.PERSISTENT_OFF, 37, "step")
        run(nx, ny, bnd, prec, lbm13.PERSISTENT_AUTO, 37, "resident")
    for bnd in (box, W.boundary(), W.cavity(T0, 0.01, 1e-4)):
        run(901, 803, bnd, prec, lbm13.PERSISTENT_ON, 5, "barrier")
torch.cuda.synchronize()
print(json.dumps(dict(launches, violations=sum(g.debug_violations() for g in lats))))
"""


def test_every_way_of_stepping_stays_inside_the_lattice(L):
    from paper_1401_0188_gb300 import build
    build.build(debug=True)
    env = dict(os.environ, LBM13_DEBUG_BUILD="1")
    r = subprocess.run([sys.executable, "-c", SCRIPT], cwd=ROOT, env=env, capture_output=True, text=True, timeout=1200)
    assert r.returncode == 0, r.stderr[-3000:]
    d = json.loads(r.stdout.strip().splitlines()[-1])
    assert d == {"step": 14, "resident": 14, "barrier": 6, "violations": 0}, d


def test_a_lattice_is_set_up_beside_a_plan_in_shared_memory(L):
    """As the solve server admits one while a round of 24 runs: 0.65 ms measured (0.45
    alone, 3.5 with a tile of the plan on every SM)."""
    import time
    import torch
    s, t = torch.cuda.Stream(), torch.cuda.Stream()
    lats = [_lattice(L, n, n, "cavity_zero_flux", 1, L.PERSISTENT_AUTO, s) for n in (64, 96, 128) * 8]
    plan = L.Plan(lats, stream=s)
    plan.step(64)
    took = []
    for _ in range(6):  # the first ones take their memory from the device
        torch.cuda.synchronize()
        end = torch.cuda.Event()
        plan.step(2000)
        end.record(s)
        time.sleep(5e-4)
        t0 = time.perf_counter()
        b = L.Lattice(128, 128, lats[0].params, lats[0].bnd, precision=1, stream=t)
        b.set_state(None, None, None, None)  # at rest
        b.residual()
        took.append(1.0 if end.query() else time.perf_counter() - t0)
        b.close()
    assert min(took) < 2e-3, took
    plan.close()


@pytest.mark.parametrize("size", [(64, 64), (187, 211), (256, 256), (360, 360), (700, 600), (901, 803)])
@pytest.mark.parametrize("precision", [0, 1])
def test_a_lattice_holds_no_more_than_the_server_counts(L, precision, size):
    from paper_1401_0188_gb300 import serving
    g = _lattice(L, *size, "cavity", precision, L.PERSISTENT_AUTO)
    g.step(64)
    g.residual()
    assert g.info()["device_bytes"] <= serving.lattice_bytes(*size, precision)
    g.close()
