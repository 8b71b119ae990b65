"""The forward model, gradient and VJP on packed real rows (two rows per complex
row, half the columns) against the FP64 oracle and against the full complex
passes, at the edges of the packing: 16 rows (fewer packed rows than a CTA
holds), bins that are their own mirrors, lengths with a factor 3, several
projections per CTA. Tolerances are the parity ones: forward 1e-5, gradients
1e-4, loss 1e-5 relative."""
import numpy as np
import pytest

from oracle import pwf_oracle as O
from paper_2503_20146_gb300 import synth as S

from _cases import blob_batch, geometry, rel_l2, to_c64, to_f32

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

FWD_TOL, GRAD_TOL, LOSS_TOL = 1e-5, 1e-4, 1e-5


@pytest.fixture(scope="module")
def pwf():
    from paper_2503_20146_gb300 import _build
    _build.build()
    from paper_2503_20146_gb300 import pwf as P
    P.load()
    return P


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.mark.parametrize("batch,ny,nx", [(1, 16, 16), (3, 16, 256), (5, 32, 16), (2, 96, 64), (1, 64, 768), (3, 128, 96),
                                         (1, 256, 1024), (1, 16, 2048), (2, 1536, 32)])
def test_packed_forward_gradient_and_vjp(pwf, batch, ny, nx):
    w = S.WORKLOADS["blob512_iotf"]
    geom = geometry(w, ny, nx)
    psi_true, t = blob_batch(w, batch, ny, nx)
    rng = np.random.default_rng(ny * 10000 + nx)
    psi, t = to_c64(0.5 * psi_true), to_c64(t * (0.8 + 0.2 * rng.random((ny, nx))))
    P64, T64 = psi.astype(np.complex128), t.astype(np.complex128)
    y = to_f32(O.intensity_batch(psi_true, T64, geom) * (1.0 + 0.05 * rng.standard_normal((batch, ny, nx))))
    cot = to_f32(rng.standard_normal((batch, ny, nx)))
    out = []
    for flag in (0, pwf.FLAG_UNPACKED_RESID):
        desc = pwf.PlanDesc(batch, ny, nx, w.pixel_m, w.wavelength_m, w.L1_m, w.L2_m, w.xcoh_m, w.ycoh_m, w.gamma,
                            w.alpha.real, w.alpha.imag, w.eta, flag)
        with pwf.Plan(desc) as plan:
            shapes = [None] if flag else list(range(pwf.pwf_plan_column_shapes(plan.handle, 6)))
            for shape in shapes:
                if shape is not None:  # asks for the packed form on a small plan
                    try:
                        pwf.pwf_plan_set_column_shape(plan.handle, 6, shape)
                    except pwf.PWFError:  # a tile wider than nx/2
                        continue
                f = plan.forward(dev(psi), dev(t))
                g, loss = plan.gradient(dev(psi), dev(t), dev(y))
                gp, gt = plan.vjp(dev(psi), dev(t), dev(cot))
                out.append([x.cpu().numpy() for x in (f, g, loss, gp, gt)])
    f_ref = O.intensity_batch(P64, T64, geom)
    g_ref, l_ref = O.gradient_batch(P64, T64, y.astype(np.float64), geom)
    gp_ref, gt_ref = O.forward_vjp_batch(P64, T64, cot.astype(np.float64), geom)
    for f, g, loss, gp, gt in out:
        assert rel_l2(f, f_ref) <= FWD_TOL
        assert rel_l2(g, g_ref) <= GRAD_TOL
        assert rel_l2(loss, l_ref) <= LOSS_TOL
        assert rel_l2(gp, gp_ref) <= GRAD_TOL
        assert rel_l2(gt, gt_ref) <= GRAD_TOL
