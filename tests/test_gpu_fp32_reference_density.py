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


@pytest.mark.parametrize("precision", [lbm.FP32_SHIFTED, lbm.FP32_CONSERVED])
@pytest.mark.parametrize("rho0", [0.9, 1.3])
def test_batch_of_mixed_reference_densities(rho0, precision):
    """One lattice with a reference density outside [1/2, 2) puts a batch on the kernel that reads each
    lattice's constants; every lattice still has the bits of its own lbm_run.  A last bit of a float64
    density decides a float32 rounding once in some 10^8 sites, hence the size."""
    require_gpu()
    params, fa, fb, want = [], [], [], []
    for j, (lx, ly, r) in enumerate([(2048, 2048, rho0), (24, 50, 3.0), (27, 63, 0.3), (30, 76, 0.7)]):
        p = lbm.Params(lx, ly, tau=0.7, gx=1e-4, rho0=r, precision=precision)
        rho, ux, uy, T = rt_fields(p, seed=40 + j)
        f = device_init(p, [t.contiguous() for t in (rho * r, ux + 0.02, uy - 0.01, T)])
        params.append(p)
        want.append(lbm.run(p, f.clone(), lbm.empty_state(p), 300).clone())
        fa.append(f)
        fb.append(lbm.empty_state(p))
    b = lbm.Batch(params, fa, fb)
    b.run(300)
    for p, got, w in zip(params, b.states(), want):
        assert torch.equal(got[:, :, :p.ly], w[:, :, :p.ly]), p.rho0
    b.close()


@pytest.mark.parametrize("precision", [lbm.FP32_SHIFTED, lbm.FP32_CONSERVED])
@pytest.mark.parametrize("mode", [lbm.BATCH_PER_STEP, lbm.BATCH_PERSISTENT])
@pytest.mark.parametrize("bc", [lbm.BC_WALLS, lbm.BC_PERIODIC_Y])
@pytest.mark.parametrize("densities", [(0.7, 1.3, 1.0), (3.0, 0.3, 1600.0), (0.9, 3.0, 1.0, 0.3)])
def test_batches_in_each_instantiation(densities, bc, mode, precision):
    """Reference densities all inside [1/2, 2), all outside, and both: the bits of the single runs."""
    require_gpu()
    params, fa, want = [], [], []
    for j, rho0 in enumerate(densities):
        p = lbm.Params(11 + 3 * j, 33 + 13 * j, tau=0.7, gx=1e-4, rho0=rho0, precision=precision, bc=bc)
        rho, ux, uy, T = rt_fields(p, seed=40 + j)
        fa.append(device_init(p, [t.contiguous() for t in (rho * rho0, ux + 0.02, uy - 0.01, T)]))
        params.append(p)
        want.append(lbm.run(p, fa[-1].clone(), lbm.empty_state(p), 5).clone())
    b = lbm.Batch(params, fa, [lbm.empty_state(p) for p in params])
    b.configure(mode, 2)
    b.run(5)
    for p, got, w in zip(params, b.states(), want):
        assert torch.equal(got[:, :, :p.ly], w[:, :, :p.ly]), p.rho0
    b.close()
