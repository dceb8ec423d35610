"""The fixed-point adjoint of a site's collision (adjoint_fix64.cuh, built for the host) against exact
rational arithmetic, over the scales of the populations and of lambda, alone and together.

Bounds, in units of 2^-K (max |lambda| 2^K is in [2^57, 2^58)): a moment carries at most half a unit of
2^(-1-K) from each of its 19 weightings, times the multiples of the velocities; the coefficients that
multiply it in a result fall as those grow, and four floors follow.  64 units of 2^-K hold an output
(the multiples, up to |v|^2 c^2 = 14, are its largest factor) and, at the density's scale 2^k, tau^2
times the site's part of dL/dtau; a few float64 roundings of the value come on top.
"""
import os
import random
import shutil
import subprocess
from fractions import Fraction as F

import pytest

from tests.test_site_fix64_host import bits, equilibrium, from_bits, model, state  # noqa: F401 (model: a fixture)

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    exe = str(tmp_path_factory.mktemp("adjoint") / "adjoint_fix64_host")
    subprocess.run([nvcc, "-std=c++17", "--expt-relaxed-constexpr", "-o", exe,
                    os.path.join(HERE, "native", "adjoint_fix64_host.cu")], check=True, capture_output=True)

    def run(lines):
        out = subprocess.run([exe], input="\n".join(lines) + "\n", capture_output=True, text=True, check=True)
        return [line.split() for line in out.stdout.splitlines()]
    return run


def collide(model, f, tau, gx, gy):  # noqa: F811
    """The collision in the numbers' own arithmetic, all of tau's uses included."""
    c, w, vx, vy = model
    c2, one = F(c * c), F(1)
    rho = sum(f)
    X = c2 * sum(a * v for a, v in zip(vx, f)) / rho
    Y = c2 * sum(a * v for a, v in zip(vy, f)) / rho
    T = (c2 * sum((a * a + b * b) * v for a, b, v in zip(vx, vy, f)) / rho - (X * X + Y * Y) / c2) / 2
    T += tau * (one - tau) * (gx * gx + gy * gy) / 2
    X, Y = X + F(c) * tau * gx, Y + F(c) * tau * gy
    return [(one - one / tau) * v + equilibrium(model, i, rho, X, Y, T, c2) / tau for i, v in enumerate(f)]


H = F(2) ** -60  # step of the central differences: the third order is below 2^-100 of the values


def exact(model, f, lam, tau, gx, gy):  # noqa: F811
    """(J^T lambda, lambda . d collide / d tau), J the collision's Jacobian."""
    f, lam, tau, gx, gy = [F(v) for v in f], [F(v) for v in lam], F(tau), F(gx), F(gy)

    def along(a, b):
        return sum(v * (x - y) for v, x, y in zip(lam, a, b)) / (2 * H)
    out = []
    for j in range(37):
        scale = f[j]
        p, m = list(f), list(f)
        p[j], m[j] = f[j] + H * scale, f[j] - H * scale
        out.append(along(collide(model, p, tau, gx, gy), collide(model, m, tau, gx, gy)) / scale)
    return out, along(collide(model, f, tau + H, gx, gy), collide(model, f, tau - H, gx, gy))


@pytest.mark.parametrize("rho,lam_scale", [
    (1.0, 1.0), (1600.0, 1.0), (1.0, 1e15), (1600.0, 1e14), (1600.0, 1e16), (16.0, 2.0 ** 54), (2.0 ** 57, 2.0 ** 54),
    (1e-250, 1e-160), (1e-250, 1e-270), (1e-250, 1e16), (2.0 ** 57, 1e-270),
])
def test_results_against_exact_arithmetic(model, probe, rho, lam_scale):  # noqa: F811
    rng = random.Random(11)
    sites = []
    for _ in range(2):
        f = state(model, rng, rho * rng.uniform(0.7, 1.0), 0.1, 0.15)
        lam = [rng.uniform(-1.0, 1.0) * lam_scale for _ in range(37)]
        sites.append((f, lam, rng.uniform(0.6, 1.5), rng.uniform(-3e-4, 3e-4), rng.uniform(-3e-4, 3e-4)))
    got = probe([" ".join([bits(t), bits(gx), bits(gy)] + [bits(v) for v in f + lam]) for f, lam, t, gx, gy in sites])
    for (f, lam, tau, gx, gy), line in zip(sites, got):
        assert line[0] == "1"
        k, K = int(line[1]), int(line[2])
        want, want_tau = exact(model, f, lam, tau, gx, gy)
        unit = F(2) ** -K
        for h, v in zip(line[4:], want):
            assert abs(F(from_bits(h)) - v) <= 64 * unit + abs(v) * F(2) ** -50
        bound = 64 * unit * F(2) ** k / F(tau) ** 2 + abs(want_tau) * F(2) ** -50 + F(2) ** -1074
        assert abs(F(from_bits(line[3])) - want_tau) <= bound, (float(want_tau), from_bits(line[3]))


@pytest.mark.parametrize("tau", [0.5 + 2.4e-10, 0.5 + 1e-6, 0.5001, 0.50024, 900.0, 1100.0, 1e5, 5e5])
def test_relaxation_times_at_both_ends(model, probe, tau):  # noqa: F811
    """Wherever the forward step takes a relaxation time in fixed point, its adjoint does."""
    rng = random.Random(12)
    f = state(model, rng, 1.0, 0.1, 0.15)
    lam = [rng.uniform(-1.0, 1.0) for _ in range(37)]
    g = 1e-4 if tau < 1.0 else 0.0
    line = probe([" ".join([bits(v) for v in [tau, g, -g] + f + lam])])[0]
    assert line[0] == "1"
    k, K = int(line[1]), int(line[2])
    want, want_tau = exact(model, f, lam, tau, g, -g)
    unit = F(2) ** -K
    for h, v in zip(line[4:], want):
        assert abs(F(from_bits(h)) - v) <= 64 * unit + abs(v) * F(2) ** -50
    assert abs(F(from_bits(line[3])) - want_tau) <= 64 * unit * F(2) ** k / F(tau) ** 2 + abs(want_tau) * F(2) ** -50
