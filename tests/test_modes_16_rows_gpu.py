"""Source-mode plans with 16 rows: one thread per column transform, so that the
mode column passes run in CTAs of half a warp. Forward, gradient, VJP and
iterations against the FP64 oracle; tolerances as for every other size."""
import numpy as np
import pytest

from oracle import pwf_oracle as O
from paper_2503_20146_gb300 import synth as S

from _cases import blob_batch, geometry, phase_rms, rel_l2, to_c64, to_f32

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

FWD_TOL, GRAD_TOL, LOSS_TOL, PHASE_TOL = 1e-5, 1e-4, 1e-5, 1e-3
SIGMA = 2.0
W2 = S.WORKLOADS["blob512_iotf"]


@pytest.fixture(scope="module")
def pwf():
    from paper_2503_20146_gb300 import _build
    _build.build()
    from paper_2503_20146_gb300 import pwf as P
    P.load()
    return P


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.mark.parametrize("K,batch,nx", [(9, 1, 16), (9, 3, 64), (25, 2, 16), (9, 2, 96), (25, 1, 2048)])
def test_sixteen_rows(pwf, K, batch, nx):
    ny = 16
    geom = geometry(W2, ny, nx)
    modes = O.source_modes(geom, K, SIGMA)
    psi, t = blob_batch(W2, batch, ny, nx)
    psi, t = to_c64(psi), to_c64(t)
    rng = np.random.default_rng(16 * nx + K)
    y = to_f32(np.clip(1.0 + 0.1 * rng.standard_normal((batch, ny, nx)), 0, None))
    gf = to_f32(rng.standard_normal((batch, ny, nx)))
    desc = pwf.PlanDesc(batch, ny, nx, geom.pixel, geom.wavelength, geom.L1, geom.L2, geom.xcoh, geom.ycoh, geom.gamma,
                        geom.alpha.real, geom.alpha.imag, geom.eta, 0, K, SIGMA)
    with pwf.Plan(desc) as plan:
        assert min(pwf.pwf_plan_column_shapes(plan.handle, m) for m in (7, 8)) >= 1
        f = plan.forward(dev(psi), dev(t)).cpu().numpy()
        g, loss = plan.gradient(dev(psi), dev(t), dev(y))
        g, loss = g.cpu().numpy(), loss.cpu().numpy()
        gp, gt = plan.vjp(dev(psi), dev(t), dev(gf))
        gp, gt = gp.cpu().numpy(), gt.cpu().numpy()
        p = torch.zeros((batch, ny, nx), dtype=torch.complex64, device="cuda")
        iters, _ = plan.solve(dev(y), dev(t), p, 5)
        p = p.cpu().numpy()
    assert list(iters) == [5] * batch
    T64 = t.astype(np.complex128)
    gt_ref = np.zeros_like(T64)
    for b in range(batch):
        P64, y64 = psi[b].astype(np.complex128), y[b].astype(np.float64)
        assert rel_l2(f[b], O.modal_intensity(P64, T64, geom, modes)) <= FWD_TOL
        ge, le = O.modal_gradient(P64, T64, y64, geom, modes)
        assert rel_l2(g[b], ge) <= GRAD_TOL and abs(loss[b] - le) <= LOSS_TOL * le
        vp, vt = O.modal_forward_vjp(P64, T64, gf[b].astype(np.float64), geom, modes)
        assert rel_l2(gp[b], vp) <= GRAD_TOL
        gt_ref += vt
        assert phase_rms(p[b], O.modal_solve(y64, T64, geom, modes, 5).psi) <= PHASE_TOL
    assert rel_l2(gt, gt_ref) <= GRAD_TOL
