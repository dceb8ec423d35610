"""The fixed-point site collision (site_fix64.cuh, built for the host) against exact rational
arithmetic, over its range, at its edges and outside it.

Bound: the float64 rounding of a result, 2^-53 of it, plus 12 units of 2^-57 at its shell's
scale 2^(k - e_s): up to 1.5 for the two products' floors and dropped low words, 5 for the at
most ten floors of 2^-58 in p, the rest for the scalars (the temperature and the velocities are
within 2^-58, and the polynomial's slopes stay below 12 in range).
"""
import os
import random
import shutil
import struct
import subprocess
from fractions import Fraction as F

import pytest

from paper_1703_04594_gb300 import lbm
from tests.gpu_util import ensure_built

HERE = os.path.dirname(os.path.abspath(__file__))
SHELL_EXP = {0: 2, 1: 3, 2: 4, 4: 6, 5: 7, 8: 9, 9: 11, 10: 11}


@pytest.fixture(scope="module")
def model():
    ensure_built()
    return lbm.model()


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    exe = str(tmp_path_factory.mktemp("site") / "site_fix64_host")
    subprocess.run([nvcc, "-std=c++17", "--expt-relaxed-constexpr", "-o", exe,
                    os.path.join(HERE, "native", "site_fix64_host.cu")], check=True, capture_output=True)

    def run(lines):
        out = subprocess.run([exe], input="\n".join(lines) + "\n", capture_output=True, text=True, check=True)
        return [line.split() for line in out.stdout.splitlines()]
    return run


def bits(v):
    return format(struct.unpack("<Q", struct.pack("<d", v))[0], "x")


def from_bits(h):
    return struct.unpack("<d", struct.pack("<Q", int(h, 16)))[0]


def equilibrium(model, i, rho, X, Y, T, c2):
    """w_i rho P_i in the numbers' own arithmetic (floats or Fractions), X = c u_x, Y = c u_y."""
    _, w, vx, vy = model
    one = type(rho)(1)
    q, t = c2 * (vx[i] ** 2 + vy[i] ** 2), T - one
    s, U = vx[i] * X + vy[i] * Y, (X * X + Y * Y) / c2
    c0 = one - U / 2 + t * (q - 2) / 2 + U * U / 8 + t * U * (4 - q) / 4 + t * t * (q * q - 8 * q + 8) / 8
    k1, k2 = one - U / 2 + t * (q - 4) / 2, one / 2 - U / 4 + t * (q - 6) / 4
    return type(rho)(w[i]) * rho * (c0 + s * k1 + s * s * k2 + s * s * s / 6 + s * s * s * s / 24)


def collided(model, f, tau, gx, gy):
    """The collision of the library's own constants: c^2, 1 / tau and 1 - 1 / tau, the shifts of
    the velocity and of the temperature are float64 numbers."""
    c, w, vx, vy = model
    c2 = F(c * c)
    om, om1 = F(1.0 / tau), F(1.0 - 1.0 / tau)
    f = [F(v) for v in f]
    rho = sum(f)
    X = c2 * sum(a * v for a, v in zip(vx, f)) / rho
    Y = c2 * sum(a * v for a, v in zip(vy, f)) / rho
    T = (c2 * sum((a * a + b * b) * v for a, b, v in zip(vx, vy, f)) / rho - (X * X + Y * Y) / c2) / 2
    T += F(tau * (1.0 - tau) * (gx * gx + gy * gy) / 2.0)
    X, Y = X + F(c * tau * gx), Y + F(c * tau * gy)
    return [om1 * v + om * equilibrium(model, i, rho, X, Y, T, c2) for i, v in enumerate(f)]


def state(model, rng, rho, u, t, off=0.02):
    ux, uy, T = rng.uniform(-u, u), rng.uniform(-u, u), 1.0 + rng.uniform(-t, t)
    c = model[0]
    return [equilibrium(model, i, rho, c * ux, c * uy, T, c * c) * (1.0 + rng.uniform(-off, off)) for i in range(37)]


@pytest.mark.parametrize("rho,u,t,taus", [
    (1.0, 0.05, 0.15, (0.6, 1.2)),          # ordinary states
    (1600.0, 0.1, 0.15, (0.55, 2.0)),       # dense
    (3e-4, 0.1, 0.15, (0.55, 2.0)),         # thin
    (1.0, 0.28, 0.38, (0.501, 30.0)),       # to the edges of the range
])
def test_results_against_exact_arithmetic(model, probe, rho, u, t, taus):
    rng = random.Random(5)
    _, _, vx, vy = model
    sites = []
    for _ in range(150):
        tau = rng.uniform(*taus)
        sites.append((state(model, rng, rho * rng.uniform(0.7, 1.4), u, t), tau, rng.uniform(-3e-4, 3e-4),
                      rng.uniform(-3e-4, 3e-4)))
    got = probe([" ".join([bits(tau), bits(gx), bits(gy)] + [bits(v) for v in f]) for f, tau, gx, gy in sites])
    inside = 0
    for (f, tau, gx, gy), line in zip(sites, got):
        if line[0] == "0":
            continue
        inside += 1
        k = int(line[1])
        for i, (h, want) in enumerate(zip(line[2:], collided(model, f, tau, gx, gy))):
            unit = F(2) ** (k - SHELL_EXP[vx[i] ** 2 + vy[i] ** 2] - 57)
            assert abs(F(from_bits(h)) - want) <= abs(want) * F(2) ** -53 + 12 * unit, (i, tau)
    assert inside >= (150 if u <= 0.1 else 60)


def test_sites_outside_the_range_are_refused(model, probe):
    rng = random.Random(6)
    base = state(model, rng, 1.0, 0.02, 0.02)
    bad = []
    for i in (0, 7, 36):
        for v in (0.0, -base[i], base[i] * 2.0 ** -12, base[i] * 16.0, float("inf"), float("nan"), 5e-324, 1e300):
            f = list(base)
            f[i] = v
            bad.append(f)
    bad.append([-v for v in base])
    bad.append([v * 1e-300 for v in base])
    c = model[0]
    bad.append([equilibrium(model, i, 1.0, c * 0.4, 0.0, 1.0, c * c) for i in range(37)])
    bad.append([equilibrium(model, i, 1.0, 0.0, 0.0, 1.5, c * c) for i in range(37)])
    head = [bits(0.8), bits(0.0), bits(-1e-4)]
    got = probe([" ".join(head + [bits(v) for v in f]) for f in bad] + [" ".join(head + [bits(v) for v in base])])
    assert [g[0] for g in got] == ["0"] * len(bad) + ["1"]
    # constants outside the formats: a forcing of tau g = 0.4
    assert probe([" ".join([bits(0.8), bits(0.5), bits(0.0)] + [bits(v) for v in base])])[0][0] == "0"


def results_or_refused(model, probe, sites):
    """Each site is refused or within the bound; returns how many were taken."""
    _, _, vx, vy = model
    got = probe([" ".join([bits(tau), bits(gx), bits(gy)] + [bits(v) for v in f]) for f, tau, gx, gy in sites])
    inside = 0
    for (f, tau, gx, gy), line in zip(sites, got):
        if line[0] == "0":
            continue
        inside += 1
        k = int(line[1])
        for i, (h, want) in enumerate(zip(line[2:], collided(model, f, tau, gx, gy))):
            unit = F(2) ** (k - SHELL_EXP[vx[i] ** 2 + vy[i] ** 2] - 57)
            assert abs(F(from_bits(h)) - want) <= abs(want) * F(2) ** -53 + 12 * unit, (i, tau)
    return inside


@pytest.mark.parametrize("above", [2.0 ** -53, 1e-15, 1e-12, 1e-10, 1.1e-10, 1.2e-10, 2.3e-10, 2.4e-10, 1e-9, 1e-6])
def test_relaxation_times_just_above_one_half(model, probe, above):
    """omega close to 2, the end of its format: from 2 - 2^-31 on its high half would round up to 2^31."""
    rng = random.Random(7)
    sites = [(state(model, rng, rng.uniform(0.7, 1.4), 0.1, 0.15), 0.5 + above, 0.0, -1e-4) for _ in range(20)]
    inside = results_or_refused(model, probe, sites)
    assert inside == (20 if above >= 1e-9 else 0 if above <= 2e-10 else inside)


def edge_site(model, rho, jx, energy):
    """Populations with f_0 just below 1/8, so that the site's scale is 1, inside their own ranges, of
    density rho, momentum (jx, 0) and sum |v|^2 f = energy up to 2^-40."""
    from scipy.optimize import linprog
    _, _, vx, vy = model
    shell = [a * a + b * b for a, b in zip(vx, vy)]
    top = [2.0 / 2 ** SHELL_EXP[s] for s in shell]
    bounds = [(0.0626, 0.1249)] + [(v * 1.05 / 256, v * 0.95) for v in top[1:]]
    sol = linprog([0.0] * 37, A_eq=[[1.0] * 37, vx, vy, shell], b_eq=[rho, jx, 0.0, energy], bounds=bounds)
    assert sol.success
    return [round(v * 2.0 ** 50) * 2.0 ** -50 for v in sol.x]


@pytest.mark.parametrize("gap", [2.0 ** -12, 2.0 ** -29, 2.0 ** -35])
@pytest.mark.parametrize("rho", [0.97, 0.98, 0.995])
def test_sums_at_the_ends_of_their_formats(model, probe, rho, gap):
    """Momentum just below 1/4 and energy just below 1/2 above that of T = 1 at the site's scale: the
    ends of the formats, where a high half would round up past them."""
    c2 = model[0] ** 2
    sites = []
    for t in (-0.3, -0.1, 0.0, 0.1):
        jx = 0.25 - gap
        sites.append((edge_site(model, rho, jx, (2.0 * (1.0 + t) * rho + c2 * jx * jx / rho) / c2), 0.8, 0.0, 0.0))
    for jx in (0.0, 0.05):
        sites.append((edge_site(model, rho, jx, 2.0 * rho / c2 + 0.5 - gap), 0.8, 0.0, 0.0))
    inside = results_or_refused(model, probe, sites)
    assert gap < 2.0 ** -12 or inside >= 4
