"""The fields and the energy of float64 states through each of their routes: the fixed-point scalars, the
fixed-point sums with float64 scalars, integer sums at the exponent of the largest population, and plain
float64 sums."""
import pytest
import torch

from paper_1703_04594_gb300 import lbm
from tests.gpu_util import require_gpu

pytestmark = pytest.mark.gpu


def fields_and_energy(p, f):
    return [t.cpu() for t in lbm.moments(p, f)], float(lbm.kinetic_energy(p, f))


def reference(f):
    """Float64 sums over populations scaled to about 1 (a power of two, exactly), and the sum of their sizes."""
    c, w, vx, vy = lbm.model()
    a, b = (torch.tensor(v, dtype=torch.float64)[:, None, None] for v in (vx, vy))
    rho, jx, jy, e = f.sum(0), c * (a * f).sum(0), c * (b * f).sum(0), c * c * ((a * a + b * b) * f).sum(0)
    ux, uy = jx / rho, jy / rho
    return [rho, ux, uy, (e / rho - ux * ux - uy * uy) / 2], f.abs().sum(0)


@pytest.mark.parametrize("power", [0, 11, -30, 55, -900, 960, -1000, 1010])
@pytest.mark.parametrize("spread,sign", [(0.1, 0.0), (0.9, 0.0), (3.0, 0.0), (0.9, 0.2), (30.0, 0.1)])
def test_fields_of_any_populations(power, spread, sign):
    """Populations w_i 2^power exp(spread n), a share of them negative: the four routes side by side.  Both
    the reference and the library carry below 37 2^-53 of sum |f| in a sum (10 times that in the energy's),
    and u and T divide by rho: 1e-13 of sum |f| / |rho| for u, 1e-12 of it for T and, squared, for what u
    adds to it."""
    require_gpu()
    p = lbm.Params(9, 70)
    g = torch.Generator().manual_seed(31)
    w = torch.tensor(lbm.model()[1], dtype=torch.float64)[:, None, None]
    f = w * torch.exp(spread * torch.randn(37, p.lx, p.ly, dtype=torch.float64, generator=g))
    f = torch.where(torch.rand(f.shape, generator=g) < sign, -f, f)
    f[:, ::2, ::3] *= 0.0 if sign else 1.0
    f[5, ::2, ::3] += 1.0                          # sites with one population beside zeros
    scaled = torch.ldexp(f, torch.tensor(power))
    scaled = torch.where(scaled.isfinite(), scaled, torch.ldexp(w, torch.tensor(power)).expand_as(f))  # e^120 2^960
    f = torch.ldexp(scaled, torch.tensor(-power))  # what subnormals left of it
    state = torch.zeros((37, p.lx, lbm.pitch(p)), dtype=torch.float64)
    state[:, :, :p.ly] = scaled
    got, ke = fields_and_energy(p, state.cuda())
    want, size = reference(f)
    # where the sums are numbers (up to sum |v|^2 |f| c^2, 15 times that of the populations)
    held = torch.ldexp(15 * size, torch.tensor(power)).isfinite()
    got, want, size = [t[held] for t in got], [t[held] for t in want], size[held]
    assert len(size) > (200 if power > 900 else 600)
    cond = size / want[0].abs()
    assert float(((torch.ldexp(got[0], torch.tensor(-power)) - want[0]).abs() / size).max()) <= 1e-13
    for a, b in zip(got[1:3], want[1:3]):
        assert float(((a - b).abs() / ((1 + b.abs()) * cond)).max()) <= 1e-13
    uu = want[1] ** 2 + want[2] ** 2
    assert float(((got[3] - want[3]).abs() / ((1 + uu + want[3].abs()) * cond)).max()) <= 1e-12
    terms = torch.ldexp(0.5 * want[0] * uu, torch.tensor(power))
    bound = torch.ldexp((0.5 * want[0].abs() * (1 + uu) * cond).sum(), torch.tensor(power))
    if abs(power) <= 960 and bool(held.all()) and bool(bound.isfinite()):
        assert abs(ke - float(terms.sum())) <= 1e-12 * float(bound)


@pytest.mark.parametrize("bad", [float("inf"), -float("inf"), float("nan"), 1e308])
def test_fields_next_to_a_population_beyond_numbers(bad):
    """One such population flags its own site and no other; a population of 1e308 is a number."""
    require_gpu()
    p = lbm.Params(5, 40)
    f = torch.zeros((37, p.lx, lbm.pitch(p)), dtype=torch.float64)
    f[:, :, :p.ly] = torch.tensor(lbm.model()[1], dtype=torch.float64)[:, None, None]
    clean = [t.cpu() for t in lbm.moments(p, f.cuda())]
    f[7, 2, 33] = bad
    got = [t.cpu() for t in lbm.moments(p, f.cuda())]
    other = torch.ones(p.lx, p.ly, dtype=torch.bool)
    other[2, 33] = False
    for a, b in zip(got, clean):
        assert torch.equal(a[other], b[other])
    if bad == 1e308:
        assert abs(float(got[0][2, 33]) / bad - 1.0) <= 1e-15
    else:
        assert not torch.isfinite(got[0][2, 33]) and torch.isnan(got[3][2, 33])
