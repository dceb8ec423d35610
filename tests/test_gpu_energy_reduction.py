"""The kinetic energy's sum of per-tile partials at the edges of its two forms: one block up to 8192
partials, a cluster of eight blocks beyond, with parts of unequal length and of less than a round of
loads."""
import pytest
import torch

from paper_1703_04594_gb300 import lbm
from tests.gpu_util import require_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [lbm.FP64, lbm.FP32_SHIFTED])
@pytest.mark.parametrize("lx,ly", [(4, 6), (32768, 6), (32769, 6), (32772, 31), (65535, 6), (3000, 710), (2049, 8192)])
def test_energy_of_many_partials(lx, ly, precision):
    """Against the sum of rho |u|^2 / 2 over the state's own fields.  Both sum n non-negative terms, each
    of a handful of roundings, in chains of at most 2^17 additions: 1e-10 of the sum is far above what
    they can differ by, and one lost or doubled partial of the up to 2^18 moves it by 1e-6 or more."""
    require_gpu()
    p = lbm.Params(lx, ly, precision=precision)
    x = torch.arange(lx, dtype=torch.float64, device="cuda")[:, None]
    y = torch.arange(ly, dtype=torch.float64, device="cuda")[None, :]
    rho = (1.0 + 0.1 * torch.cos(0.01 * x + 0.02 * y)).contiguous()
    ux = (0.05 + 0.01 * torch.sin(0.03 * x) + 0.0 * y).contiguous()
    uy = (0.04 * torch.ones_like(rho)).contiguous()
    f = lbm.empty_state(p)
    lbm.init(p, rho, ux, uy, torch.ones_like(rho), f)
    r, u, v, _ = lbm.moments(p, f)
    want = float((0.5 * r * (u * u + v * v)).sum())
    for _ in range(3):
        assert abs(float(lbm.kinetic_energy(p, f)) - want) <= 1e-10 * want
    assert float(lbm.kinetic_energy_noalloc(p, f)) == float(lbm.kinetic_energy(p, f))
