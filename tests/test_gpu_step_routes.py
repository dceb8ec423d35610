"""The fixed-point routes of the float64 step and its adjoint.

The fused float64 step (fixed-point collision in range, float64 elsewhere) against the separate
kernels (float64 throughout), over sizes that give every block and strip shape, both relaxation
signs, both y boundaries, and states of which some sites leave the fixed-point range."""
import pytest
import torch

from oracle import lbm as OL
from paper_1703_04594_gb300 import lbm
from tests.gpu_util import device_init, require_gpu, rt_fields, to_host
from tests.test_gpu_adjoint import oracle_vjp, reach_max

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
    # errors on the scale of the population's shell, w_i rho (an over-relaxed population may itself
    # cancel to nothing): a float64 collision's stays below ~1e-13 of it
    w = torch.tensor(lbm.model()[1], dtype=torch.float64, device="cuda")[:, None, None]
    assert float(((a - b).abs() / (w * b.sum(0))).max()) <= 2e-12
    assert bool((got[:, :, ly:] == -7.0).all())        # the padding is not written


@pytest.mark.parametrize("lx,ly", [(5, 31), (4, 32), (7, 33), (6, 97), (4, 161), (5, 64)])
@pytest.mark.parametrize("bc", [lbm.BC_WALLS, lbm.BC_PERIODIC_Y])
@pytest.mark.parametrize("tau,drift,heat,scale", [(0.7, 0.02, 1.0, 1.0), (1.4, 0.2, 1.25, 1e-9), (0.9, 0.28, 1.3, 1e3),
                                                  (0.8, 0.02, 1.0, 1e20), (0.8, 0.02, 1.0, 1e-290)])
def test_adjoint_step_on_both_routes(lx, ly, bc, tau, drift, heat, scale):
    """The adjoint step against autograd through the oracle's step, with sites on both sides of the
    fixed-point range (speeds and temperatures beyond it, lambda above and below its block range),
    over sizes that give every block and strip shape.  The bar is that of the adjoint's own
    per-element test, 1e-13 of the largest lambda within reach."""
    require_gpu()
    p = lbm.Params(lx, ly, tau=tau, gx=1e-4, gy=-2e-4, bc=bc)
    rho, ux, uy, T = rt_fields(p, seed=5)
    x = torch.arange(lx, dtype=torch.float64)[:, None]
    f = device_init(p, [t.contiguous() for t in (rho, ux + drift * (1 + 0.3 * torch.cos(x)), uy, T * heat)])
    g = torch.Generator().manual_seed(17)
    lam = torch.randn(37, lx, ly, dtype=torch.float64, generator=g)
    lam_dev = torch.zeros_like(f)
    lam_dev[:, :, :ly] = lam.cuda() * scale
    lam_n = torch.full_like(f, -7.0)
    dtau = torch.zeros((), dtype=torch.float64, device="cuda")
    lbm.adjoint_step(p, f, lam_dev, lam_n, dtau, lbm.adjoint_work(p))
    want, want_tau = oracle_vjp(p, to_host(p, f), lam)
    got = to_host(p, lam_n) / scale
    assert float(((got - want).abs() / reach_max(lam.abs().amax(0), bc)[None]).max()) <= 1e-13
    assert abs(float(dtau) / scale - want_tau) <= 1e-10 * max(abs(want_tau), float(lam.abs().sum()) * 1e-3)
    assert bool((lam_n[:, :, ly:] == -7.0).all())


def test_adjoint_of_zero_is_zero():
    require_gpu()
    p = lbm.Params(6, 97, tau=0.7, gx=1e-4)
    f = device_init(p, rt_fields(p, seed=5))
    lam = torch.zeros_like(f)
    lam_n = torch.full_like(f, 3.0)
    dtau = torch.zeros((), dtype=torch.float64, device="cuda")
    lbm.adjoint_step(p, f, lam, lam_n, dtau, lbm.adjoint_work(p))
    assert bool((lam_n[:, :, :97] == 0).all()) and float(dtau) == 0.0


@pytest.mark.parametrize("lx,ly", [(4, 6), (5, 33), (9, 64), (70, 131)])
@pytest.mark.parametrize("rho0", [1.0, 1600.0, 1e-3])
def test_initial_state_and_fields_on_both_routes(lx, ly, rho0):
    """lbm_init, lbm_moments and lbm_kinetic_energy on fields of which some leave the fixed-point range
    (|u| to 0.45, T from 0.5 to 1.5): the state against the oracle's equilibrium at 1e-13 of its
    shell's scale, the fields of a state back at 1e-12 (the parity tests' bar)."""
    require_gpu()
    p = lbm.Params(lx, ly)
    g = torch.Generator().manual_seed(23)
    rho = rho0 * (0.5 + torch.rand(lx, ly, dtype=torch.float64, generator=g))
    ux, uy = ((torch.rand(2, lx, ly, dtype=torch.float64, generator=g) - 0.5) * 0.9).unbind(0)
    T = 0.5 + torch.rand(lx, ly, dtype=torch.float64, generator=g)
    fields = [t.contiguous() for t in (rho, ux, uy, T)]
    f = device_init(p, fields)
    host = to_host(p, f)
    w = torch.tensor(lbm.model()[1], dtype=torch.float64)[:, None, None]
    assert float(((host - OL.init_equilibrium(*fields)).abs() / (w * rho)).max()) <= 1e-13
    want = OL.fields(host)
    for a, b in zip(lbm.moments(p, f), want):
        assert float((a.cpu() - b).abs().max()) <= 1e-12 * float(b.abs().max())
    ke = float(OL.kinetic_energy(host))
    assert abs(float(lbm.kinetic_energy(p, f)) - ke) <= 1e-12 * ke


@pytest.mark.parametrize("lx,ly", [(4, 6), (5, 33), (70, 131)])
@pytest.mark.parametrize("scale,wide", [(1.0, 0.1), (1e-200, 0.1), (3e5, 0.9)])
def test_gradient_of_the_initial_state_on_both_routes(lx, ly, scale, wide):
    """lbm_init_adjoint against reverse mode through the oracle's equilibrium, with fields inside the
    fixed-point range (wide = 0.1) and on both sides of it: 1e-13 of what a field's term can reach
    (sum_i |lambda_i| w_i times the density where the field is not the density, times 40)."""
    require_gpu()
    p = lbm.Params(lx, ly)
    g = torch.Generator().manual_seed(29)
    rho = 0.5 + torch.rand(lx, ly, dtype=torch.float64, generator=g)
    ux, uy = ((torch.rand(2, lx, ly, dtype=torch.float64, generator=g) - 0.5) * wide).unbind(0)
    T = 1.0 + (torch.rand(lx, ly, dtype=torch.float64, generator=g) - 0.5) * wide
    fields = [t.contiguous().requires_grad_() for t in (rho, ux, uy, T)]
    lam = torch.randn(37, lx, ly, dtype=torch.float64, generator=g)
    lam[:, 1, 2] = 0.0
    lam_dev = lbm.empty_state(p)
    lam_dev[:, :, :ly] = lam.cuda() * scale
    want = torch.autograd.grad((OL.init_equilibrium(*fields) * lam).sum(), fields)
    got = lbm.init_adjoint(p, *[t.detach().cuda() for t in fields], lam_dev)
    reach = 40.0 * (lam.abs() * torch.tensor(lbm.model()[1], dtype=torch.float64)[:, None, None]).sum(0) * rho.clamp(min=1.0)
    for a, b in zip(got, want):
        assert float(((a.cpu() / scale - b).abs() - 1e-13 * reach).max()) <= 0.0
        assert float(a[1, 2]) == 0.0


@pytest.mark.parametrize("precision", [lbm.FP64, lbm.FP32_SHIFTED])
@pytest.mark.parametrize("lx", [5, 6, 131070, 131071])
def test_columns_on_both_sides_of_the_block_width_rule(lx, precision):
    """Blocks of two columns up to lx = 131070, of four beyond: a state uniform in x stays so, and its
    columns are those of a small lattice, bit for bit."""
    require_gpu()
    small = lbm.Params(4, 6, tau=0.8, gx=1e-4, precision=precision)
    rho, ux, uy, T = rt_fields(small, seed=3)
    fields = [t[:1].expand(4, 6).contiguous() for t in (rho, ux, uy, T)]
    f = device_init(small, fields)
    p = lbm.Params(lx, 6, tau=0.8, gx=1e-4, precision=precision)
    wide = lbm.empty_state(p)
    wide[:, :, :6] = f[:, :1, :6]
    out, want = lbm.empty_state(p), lbm.empty_state(small)
    lbm.step(small, f, want)
    lbm.step(p, wide, out)
    assert torch.equal(out[:, :, :6], want[:, :1, :6].expand(37, lx, 6))


@pytest.mark.parametrize("rho0,scale", [(1600.0, 1e14), (1600.0, 1e16), (16.0, 2.0 ** 55), (1e-250, 1e-270), (1e-250, 1e3)])
def test_adjoint_step_at_large_and_small_scales_together(rho0, scale):
    """lambda and the density both far from 1: the step is linear in lambda and its part of dL/dtau in the
    density too, so both follow from the oracle's at 1 (bars as above)."""
    require_gpu()
    p = lbm.Params(6, 97, tau=0.7, gx=1e-4, gy=-2e-4)
    rho, ux, uy, T = rt_fields(p, seed=5)
    lam = torch.randn(37, p.lx, p.ly, dtype=torch.float64, generator=torch.Generator().manual_seed(17))
    one = device_init(p, (rho, ux, uy, T))
    want, want_tau = oracle_vjp(p, to_host(p, one), lam)
    f = device_init(p, (rho * rho0, ux, uy, T))
    lam_dev = torch.zeros_like(f)
    lam_dev[:, :, :p.ly] = lam.cuda() * scale
    lam_n = torch.zeros_like(f)
    dtau = torch.zeros((), dtype=torch.float64, device="cuda")
    lbm.adjoint_step(p, f, lam_dev, lam_n, dtau, lbm.adjoint_work(p))
    got = to_host(p, lam_n) / scale
    assert float(((got - want).abs() / reach_max(lam.abs().amax(0), p.bc)[None]).max()) <= 1e-13
    reach = max(abs(want_tau), float(lam.abs().sum()) * 1e-3)
    assert abs(float(dtau) - want_tau * scale * rho0) <= 1e-10 * reach * scale * rho0


@pytest.mark.parametrize("lx,ly", [(4, 6), (5, 31), (7, 33), (6, 97)])
@pytest.mark.parametrize("bc", [lbm.BC_WALLS, lbm.BC_PERIODIC_Y])
@pytest.mark.parametrize("hot", [False, True])
def test_strips_collided_in_float64(lx, ly, bc, hot):
    """A lattice whose forcing is outside the fixed-point formats, and one with every second column too
    hot for them, against the separate kernels (the bar above); the same lattices in a batch, in both
    modes, have the same bits."""
    require_gpu()
    p = lbm.Params(lx, ly, tau=0.8, gx=0.0 if hot else 0.2, gy=-2e-4, bc=bc)
    rho, ux, uy, T = rt_fields(p, seed=3)
    if hot:
        T = T + 0.5 * (torch.arange(lx, dtype=torch.float64)[:, None] % 2)
    f = device_init(p, [t.contiguous() for t in (rho, ux, uy, T)])
    tmp, want, got = lbm.empty_state(p), lbm.empty_state(p), lbm.empty_state(p)
    lbm.propagate(p, f, tmp)
    lbm.bc(p, f, tmp)
    lbm.collide(p, tmp, want)
    lbm.step(p, f, got)
    a, b = got[:, :, :ly], want[:, :, :ly]
    w = torch.tensor(lbm.model()[1], dtype=torch.float64, device="cuda")[:, None, None]
    assert float(((a - b).abs() / (w * b.sum(0).abs())).max()) <= 2e-12
    for mode in (lbm.BATCH_PER_STEP, lbm.BATCH_PERSISTENT):
        batch = lbm.Batch([p], [f.clone()], [lbm.empty_state(p)])
        batch.configure(mode, 2)
        batch.run(1)
        assert torch.equal(batch.states()[0][:, :, :ly], a)
        batch.close()


@pytest.mark.parametrize("lx,ly", [(4, 6), (5, 33), (7, 97)])
@pytest.mark.parametrize("bc", [lbm.BC_WALLS, lbm.BC_PERIODIC_Y])
def test_adjoint_of_a_lattice_outside_the_formats(lx, ly, bc):
    """A forcing outside the fixed-point formats, so that every site is taken in float64, from the first
    gather (the bar above)."""
    require_gpu()
    p = lbm.Params(lx, ly, tau=0.8, gx=0.2, gy=-2e-4, bc=bc)
    f = device_init(p, rt_fields(p, seed=5))
    lam = torch.randn(37, lx, ly, dtype=torch.float64, generator=torch.Generator().manual_seed(17))
    lam_dev = torch.zeros_like(f)
    lam_dev[:, :, :ly] = lam.cuda()
    lam_n = torch.zeros_like(f)
    dtau = torch.zeros((), dtype=torch.float64, device="cuda")
    lbm.adjoint_step(p, f, lam_dev, lam_n, dtau, lbm.adjoint_work(p))
    want, want_tau = oracle_vjp(p, to_host(p, f), lam)
    assert float(((to_host(p, lam_n) - want).abs() / reach_max(lam.abs().amax(0), bc)[None]).max()) <= 1e-13
    assert abs(float(dtau) - want_tau) <= 1e-10 * max(abs(want_tau), float(lam.abs().sum()) * 1e-3)
