"""The FP32 forms over reference densities on both sides of the unscaled range (1/2 to 2), and the
compensated sums at their walls."""
import pytest
import torch

from oracle import lbm as OL
from paper_1703_04594_gb300 import lbm
from tests.gpu_util import device_init, field_errors, oracle_params, require_gpu, rt_fields, to_host

pytestmark = pytest.mark.gpu


def params(bc, rho0, precision, lx=9, ly=70):
    return lbm.Params(lx, ly, tau=0.8, gx=1e-4, gy=-2e-4, rho0=rho0, precision=precision, bc=bc)


@pytest.mark.parametrize("precision", [lbm.FP32_SHIFTED, lbm.FP32_CONSERVED])
@pytest.mark.parametrize("bc", [lbm.BC_WALLS, lbm.BC_PERIODIC_Y])
@pytest.mark.parametrize("rho0", [1.0, 0.7, 0.3, 1e-6, 1.99, 2.5])
def test_steps_at_every_reference_density(rho0, bc, precision):
    """Three steps of a state at the reference density: the fields within 1e-5 (the form's bar), plus,
    for the conserved form, the 2^-36 to which it sums each of its 37 outputs in each step."""
    require_gpu()
    p = params(bc, rho0, precision)
    rho, ux, uy, T = rt_fields(p, seed=9)
    fields = [(rho * rho0).contiguous(), ux, uy, T]
    op = oracle_params(p)
    host = OL.init_equilibrium(*fields)
    for _ in range(3):
        host = OL.step(host, op)
    got = [t.cpu() for t in lbm.moments(p, lbm.run(p, device_init(p, fields), lbm.empty_state(p), 3))]
    want = list(OL.fields(host))
    got[0], want[0] = got[0] / rho0, want[0] / rho0
    err = field_errors(got, want)
    tol = 1e-5 + (3 * 37 * 2.0 ** -36 / rho0 if precision == lbm.FP32_CONSERVED else 0.0)
    assert max(err[k] for k in ("rho_max", "rho_rms", "T_max", "T_rms", "u_max_cs")) <= tol, err


@pytest.mark.parametrize("ly", [6, 31, 32, 70])
def test_wall_sums_beyond_the_storage_range(ly):
    """Two populations that leave through the bottom wall enter nothing but its density: 8.5 and 0
    (beyond the storage range) give the step that 4.25 and 4.25 give, to float32 rounding."""
    require_gpu()
    p = params(lbm.BC_WALLS, 1.0, lbm.FP32_SHIFTED, 9, ly)
    vy = lbm.model()[3]
    down = [i for i in range(37) if vy[i] == -3][:2]
    f = device_init(p, rt_fields(p, seed=9))
    out = []
    for a, b in ((8.5, 0.0), (4.25, 4.25)):
        g = f.clone()
        g[down[0], 4, 0], g[down[1], 4, 0] = a, b
        o = lbm.empty_state(p)
        lbm.step(p, g, o)
        out.append(o[:, :, :ly].double())
    assert bool(torch.isfinite(out[0]).all())
    assert float((out[0] - out[1]).abs().max()) <= 1e-5 * float(out[1].abs().max())
