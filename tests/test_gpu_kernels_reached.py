"""The bounded wait of stepping from shared memory, made to run out."""
import numpy as np
import pytest

from paper_1401_0188_gb300 import pstar as product_pstar
from paper_1401_0188_gb300 import workloads as W

pytestmark = pytest.mark.gpu


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

