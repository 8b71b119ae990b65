"""PWF_FLAG_CHECK_FINITE names the first pass with a bad output on the packed
route too (a plan of 2^20 pixels): a NaN count first shows in the residual of the
gradient, a NaN cotangent in its transform, and an intensity whose row sums are
finite and whose column sums are not in the IOTF filter."""
import numpy as np
import pytest

from paper_2503_20146_gb300 import synth as S

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

BATCH, N = 64, 128
W = S.WORKLOADS["blob512_iotf"]


@pytest.fixture(scope="module")
def pwf():
    from paper_2503_20146_gb300 import _build
    _build.build()
    from paper_2503_20146_gb300 import pwf as P
    P.load()
    return P


@pytest.mark.parametrize("where,first", [("y", "row_resid_pk"), ("cotangent", "row_real_fft_pk"), ("overflow", "col_iotf_pk"),
                                         ("nothing", None)])
def test_first_bad_pass(pwf, where, first):
    shape = (BATCH, N, N)
    psi = torch.zeros(shape, dtype=torch.complex64, device="cuda")
    t = torch.ones((N, N), dtype=torch.complex64, device="cuda")
    real = torch.ones(shape, device="cuda")
    if where in ("y", "cotangent"):
        real[BATCH - 1, N - 1, 3] = float("nan")
    elif where == "overflow":
        psi.real.fill_(40.5)  # |exp psi|^2 = 1.5e35: 128 of them add up to 1.9e37, 128 x 128 to more than FP32 holds
    desc = pwf.PlanDesc(BATCH, N, N, W.pixel_m, W.wavelength_m, W.L1_m, W.L2_m, W.xcoh_m, W.ycoh_m, W.gamma, W.alpha.real,
                        W.alpha.imag, W.eta, pwf.FLAG_CHECK_FINITE)
    with pwf.Plan(desc) as plan:
        state = pwf.pwf_state_create(plan.handle)
        try:
            if where in ("y", "nothing"):
                plan.gradient(psi, t, real)
            if where in ("cotangent", "nothing"):
                plan.vjp(psi, t, real)
            if where in ("overflow", "nothing"):
                plan.forward(psi, t)
            if first is None:
                pwf.pwf_state_read(plan.handle, state, BATCH)
            else:
                with pytest.raises(pwf.PWFError) as e:
                    pwf.pwf_state_read(plan.handle, state, BATCH)
                assert e.value.status == 5 and f"pass {first})" in str(e.value), str(e.value)
        finally:
            pwf.pwf_state_destroy(state)
