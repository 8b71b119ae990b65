"""Which plans take the packed real passes in forward model, gradient and VJP
(two real rows per complex row, half the columns), and that they compute the
same there. The route shows in the bits: a plan on the packed route differs from
one with PWF_FLAG_UNPACKED_RESID by rounding, a plan off it does not differ at
all (both untuned, so on the same column shapes).

From 2^20 pixels on, with a packed shape of the column length whose tile
divides nx / 2; below, choosing the shape of the solver's packed residual pass
leaves the other calls as they are. Tolerances are the parity ones."""
import numpy as np
import pytest

from oracle import pwf_oracle as O
from paper_2503_20146_gb300 import synth as S

from _cases import blob_batch, geometry, rel_l2, to_c64, to_f32

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

FWD_TOL, GRAD_TOL, LOSS_TOL = 1e-5, 1e-4, 1e-5
W = S.WORKLOADS["blob512_iotf"]


@pytest.fixture(scope="module")
def pwf():
    from paper_2503_20146_gb300 import _build
    _build.build()
    from paper_2503_20146_gb300 import pwf as P
    P.load()
    return P


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def plan_of(P, batch, ny, nx, flags):
    return P.Plan(P.PlanDesc(batch, ny, nx, W.pixel_m, W.wavelength_m, W.L1_m, W.L2_m, W.xcoh_m, W.ycoh_m, W.gamma,
                             W.alpha.real, W.alpha.imag, W.eta, flags))


def calls(plan, psi, t, y, cot):
    g, loss = plan.gradient(psi, t, y)
    gp, gt = plan.vjp(psi, t, cot)
    return [v.cpu().numpy() for v in (plan.forward(psi, t), g, loss, gp, gt)]


class Case:
    """A few different projections, repeated over the batch."""

    def __init__(self, batch, ny, nx):
        self.geom, self.which = geometry(W, ny, nx), np.arange(batch) % min(batch, 3)
        n = int(self.which.max()) + 1
        psi_true, t = blob_batch(W, n, ny, nx)
        rng = np.random.default_rng(ny * 10000 + nx)
        self.psi, self.t = to_c64(0.5 * psi_true), to_c64(t * (0.8 + 0.2 * rng.random((ny, nx))))
        self.y = to_f32(O.intensity_batch(psi_true, self.t.astype(np.complex128), self.geom) *
                        (1.0 + 0.05 * rng.standard_normal((n, ny, nx))))
        self.cot = to_f32(rng.standard_normal((n, ny, nx)))

    def inputs(self):
        return dev(self.psi[self.which]), dev(self.t), dev(self.y[self.which]), dev(self.cot[self.which])

    def oracle(self):
        P, T = self.psi.astype(np.complex128), self.t.astype(np.complex128)
        g, loss = O.gradient_batch(P, T, self.y.astype(np.float64), self.geom)
        vjp = [O.forward_vjp_batch(P[k:k + 1], T, self.cot[k:k + 1].astype(np.float64), self.geom) for k in range(len(P))]
        counts = np.bincount(self.which)
        return (O.intensity_batch(P, T, self.geom), g, loss, np.concatenate([v[0] for v in vjp]),
                sum(c * v[1] for c, v in zip(counts, vjp)))


# the smallest and largest column length with packed shapes, the narrowest and
# widest rows, lengths with a factor 3, several projections per wave
PACKED = [(1024, 32, 32), (342, 96, 32), (1024, 64, 16), (512, 128, 16), (171, 64, 96), (64, 128, 128), (2, 256, 2048),
          (1, 1024, 1024), (2, 1536, 512), (1, 2048, 768), (3, 768, 768)]


@pytest.mark.parametrize("batch,ny,nx", PACKED)
def test_packed_plans(pwf, batch, ny, nx):
    case = Case(batch, ny, nx)
    args, ref = case.inputs(), case.oracle()
    with plan_of(pwf, batch, ny, nx, pwf.FLAG_NO_TUNE | pwf.FLAG_UNPACKED_RESID) as plan:
        unpacked = calls(plan, *args)
    ran = 0
    with plan_of(pwf, batch, ny, nx, pwf.FLAG_NO_TUNE) as plan:
        for shape in range(pwf.pwf_plan_column_shapes(plan.handle, 6)):
            try:
                pwf.pwf_plan_set_column_shape(plan.handle, 6, shape)
            except pwf.PWFError:  # a tile wider than nx / 2
                continue
            out = calls(plan, *args)
            ran += 1
            assert all(not np.array_equal(a, b) for k, (a, b) in enumerate(zip(out, unpacked)) if k != 2)
            for k, tol in enumerate((FWD_TOL, GRAD_TOL, LOSS_TOL, GRAD_TOL)):
                for b in {0, batch // 2, batch - 1}:
                    assert rel_l2(out[k][b], ref[k][case.which[b]]) <= tol, (shape, k, b)
                assert rel_l2(out[k], unpacked[k]) <= 2 * tol, (shape, k)
            assert rel_l2(out[4], ref[4]) <= GRAD_TOL, shape
    assert ran >= 1


# 16 rows have no packed shape, and of 32 rows only one that is as wide as nx
UNPACKED = [(4096, 16, 16), (512, 16, 128), (2048, 32, 16), (3584, 96, 16)]


@pytest.mark.parametrize("batch,ny,nx", UNPACKED)
def test_plans_without_a_packed_shape_that_fits(pwf, batch, ny, nx):
    case = Case(batch, ny, nx)
    args, ref = case.inputs(), case.oracle()
    out = []
    for flag in (0, pwf.FLAG_UNPACKED_RESID):
        with plan_of(pwf, batch, ny, nx, pwf.FLAG_NO_TUNE | flag) as plan:
            out.append(calls(plan, *args))
    assert all(np.array_equal(a, b) for k, (a, b) in enumerate(zip(*out)) if k != 2)  # the loss is summed in any order
    assert rel_l2(out[0][0][-1], ref[0][case.which[-1]]) <= FWD_TOL
    assert rel_l2(out[0][4], ref[4]) <= GRAD_TOL


@pytest.mark.parametrize("batch,ny,nx", [(1, 128, 128), (9, 96, 768), (1, 1024, 512)])
def test_a_shape_of_the_residual_pass_changes_no_other_call(pwf, batch, ny, nx):
    args = Case(batch, ny, nx).inputs()
    with plan_of(pwf, batch, ny, nx, pwf.FLAG_NO_TUNE) as plan:
        before = calls(plan, *args)
        pwf.pwf_plan_set_column_shape(plan.handle, 6, pwf.pwf_plan_column_shapes(plan.handle, 6) - 1)
        after = calls(plan, *args)
    assert all(np.array_equal(a, b) for k, (a, b) in enumerate(zip(before, after)) if k != 2)
