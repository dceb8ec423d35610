"""The fused float64 step (fixed-point collision in range, float64 elsewhere) against the separate
kernels (float64 throughout), over sizes that give every block and strip shape, both relaxation
signs, both y boundaries, and states of which some sites leave the fixed-point range."""
import pytest
import torch

from paper_1703_04594_gb300 import lbm
from tests.gpu_util import device_init, require_gpu, rt_fields

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lx,ly", [(4, 6), (5, 31), (4, 32), (7, 33), (6, 35), (5, 64), (9, 95), (5, 97), (4, 128),
                                   (6, 161), (5, 321), (300, 6)])
@pytest.mark.parametrize("bc", [lbm.BC_WALLS, lbm.BC_PERIODIC_Y])
@pytest.mark.parametrize("tau,drift,hot", [(0.7, 0.03, 0.0), (1.4, 0.15, 0.2), (0.9, 0.3, 0.1)])
def test_fused_step_equals_the_separate_kernels(lx, ly, bc, tau, drift, hot):
    require_gpu()
    p = lbm.Params(lx, ly, tau=tau, gx=1e-4, gy=-2e-4, bc=bc)
    rho, ux, uy, T = rt_fields(p, seed=3)
    x = torch.arange(lx, dtype=torch.float64)[:, None]
    fields = (rho, ux + drift * torch.cos(x), uy - drift / 2, T + hot * torch.sin(x))
    f = device_init(p, [t.contiguous() for t in fields])
    tmp = lbm.empty_state(p)
    want = lbm.empty_state(p)
    lbm.propagate(p, f, tmp)
    lbm.bc(p, f, tmp)
    lbm.collide(p, tmp, want)
    got = torch.full_like(f, -7.0)
    lbm.step(p, f, got)
    a, b = got[:, :, :ly], want[:, :, :ly]
    # both round every population within a few units of its shell's scale: the populations of
    # these states stay above a hundredth of it, and a float64 collision's error is ~1e-14 of it
    assert float(((a - b).abs() / b.abs().clamp_min(1e-7)).max()) <= 2e-12
    assert bool((got[:, :, ly:] == -7.0).all())        # the padding is not written
