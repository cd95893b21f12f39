"""The integer collision of the FP64 step (csrc/lbm13_fixed.cuh) on the host, at the
states that flows hold: density, temperature and velocity deviations of very
different sizes, where the rest population is 30 times the diagonals or a thousandth
of the unit links.  Its error against 113 bits is no larger than that of the FP64
collision, mirrored nodes collide to mirrored populations bit for bit, and nodes at
the ends of its range stay inside 63 bits."""
import numpy as np
import pytest

import test_host_fixed as H
from oracle import oracle as O
from paper_1401_0188_gb300 import lbm13, params as P
from paper_1401_0188_gb300 import workloads as W

lib = H.lib  # the compiled harness (a module fixture)
Q = 13
# what mirroring x, mirroring y and turning by half a turn make of the links
MIRRORS = {"x": [0, 3, 2, 1, 4, 6, 5, 8, 7, 11, 10, 9, 12], "y": [0, 1, 4, 3, 2, 8, 7, 6, 5, 9, 12, 11, 10],
           "xy": [0, 3, 4, 1, 2, 7, 8, 5, 6, 11, 12, 9, 10]}
# amplitudes of density, velocity and temperature
SIZES = {"mixed": (2e-3, 1e-2, 2e-3), "density": (1e-2, 1e-4, 0.0), "temperature": (0.0, 1e-4, 5e-3),
         "slow": (1e-2, 1e-6, 5e-3), "fast": (1e-5, 1e-2, 1e-5), "flow": (1e-4, 1e-2, 1e-4), "faint": (1e-6, 1e-6, 1e-6)}


def _states(p, sizes, n, rng, noise):
    """Equilibrium deviations, and `noise` of the largest amplitude on every link."""
    M, D, _ = O.basis()
    st, c = lbm13.lbm13_derive(p)
    assert st == 0
    R, u, v, dT = (a * rng.standard_normal(n) for a in (sizes[0], sizes[1], sizes[1], sizes[2]))
    rho, T = 1 + R, P.rest_temperature(p) + dT
    jx, jy = rho * u, rho * v
    dE = rho * (26 * T - 28) - p["E0"] + 13 * rho * (u * u + v * v)
    Qe = p["c1"] + c[2] * rho + c[3] * (p["E0"] + dE)
    Re = c[5] + c[4] * rho + p["k2"] * (p["E0"] + dE)
    m = np.array([R, dE, c[6] * R + p["c_epsE"] * dE, p["c_vpi_rho"] * R + p["c_vpi_E"] * dE, jx, jy, jx * Qe, jy * Qe,
                  jx * Re, jy * Re, (jx * jx - jy * jy) / rho, jx * jy / rho, 0 * R])
    w = np.asarray(c[22:22 + Q])
    return (m / D[:, None]).T @ M + noise * max(sizes) * w * rng.standard_normal((n, Q))


@pytest.mark.parametrize("noise", [1e-3, 0.05])
@pytest.mark.parametrize("bound", ["plain", "buoyancy"])
@pytest.mark.parametrize("sizes", list(SIZES))
@pytest.mark.parametrize("params", ["pstar", "heat", "high_pr"])
def test_integer_collision_is_no_less_exact_than_fp64_at_flow_states(lib, params, sizes, bound, noise):
    p = H.PARAMS[params]()
    f = _states(p, SIZES[sizes], 4000, np.random.default_rng(11), noise)
    on, taken, (fi, fp, whole, ei, ep) = H._run(lib, p, H.BOUNDS[bound], f)
    assert on == 1 and taken.all()
    rms = lambda e: np.sqrt(np.mean(e ** 2, axis=0))  # noqa: E731
    assert np.linalg.norm(rms(ei)) <= np.linalg.norm(rms(ep)), (rms(ei), rms(ep))
    # of each population: 4000 nodes estimate an rms to 1.1%; those whose error in
    # FP64 is little more than the last rounding have at most a quarter more
    assert (rms(ei) <= 1.25 * rms(ep)).all(), rms(ei) / rms(ep)


@pytest.mark.parametrize("mirror", list(MIRRORS))
@pytest.mark.parametrize("bound", list(H.BOUNDS))
def test_mirrored_nodes_collide_to_mirrored_populations(lib, bound, mirror):
    b = H.BOUNDS[bound]
    m = MIRRORS[mirror]
    image = dict(b, gx=b["gx"] * (-1 if "x" in mirror else 1), gy=b["gy"] * (-1 if "y" in mirror else 1))
    rng = np.random.default_rng(2)
    p = H.PARAMS["pstar"]()
    f = np.concatenate([_states(p, s, 2000, rng, 1e-3) for s in SIZES.values()] + [H._states("even", 2000, rng)])
    # few significant bits: sums that end in halves are common
    g = f.copy()
    g[::2] = np.float32(g[::2])
    g[1::4] = np.round(g[1::4] * 2.0 ** 20) * 2.0 ** -20
    for x in (f, g):
        a = H._run(lib, p, b, x)
        c = H._run(lib, p, image, x[:, m])
        assert np.array_equal(a[1], c[1])
        assert np.array_equal(a[2][2][:, m], c[2][2])   # the whole collision
        assert np.array_equal(a[2][1][:, m], c[2][1])   # the FP64 one it replaces


@pytest.mark.parametrize("bound", list(H.BOUNDS))
@pytest.mark.parametrize("params", list(H.PARAMS))
def test_nodes_at_the_ends_of_the_range_stay_inside_63_bits(lib, params, bound):
    rng = np.random.default_rng(4)
    n = 20000
    top = 2.0 ** -5 * (1 - 2.0 ** -53)
    f = top * rng.choice([-1.0, 1.0], (n, Q))
    # the rest population up to 2^5 times the others, the others at most at the top;
    # the shell sums from all of one sign down to exact opposites
    f[:, 1:] *= 2.0 ** -rng.integers(0, 6, (n, 1)).astype(float)
    f[::3, 0] *= 2.0 ** -rng.integers(0, 40, len(f[::3])).astype(float)
    f[1::3, 3:5] = -f[1::3, 1:3]
    f[1::3, 7:9] = -f[1::3, 5:7]
    f[2::3, 11:] = -f[2::3, 9:11]
    f *= 2.0 ** -rng.choice([0, 1, 20], (n, 1)).astype(float)
    on, taken, (fi, fp, whole, ei, ep) = H._run(lib, H.PARAMS[params](), H.BOUNDS[bound], f)
    assert on == 1 and taken.mean() > 0.6
    scale = np.maximum(np.abs(f).max(axis=1), np.abs(fp).max(axis=1))[taken, None] * 2.0 ** -53
    # a sum beyond 63 bits would be off by 2^4 populations, 2^57 of these units
    assert np.abs(ei[taken] / scale).max() <= 4.0
