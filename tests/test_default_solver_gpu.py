"""Which solver a plan takes when none is asked for: the cluster-resident one for
square 128^2 plans of one wave of clusters, the graph for every other plan, 256^2
among them (which the cluster solver serves on request)."""
import pytest

from paper_2503_20146_gb300 import synth as S

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

W = S.WORKLOADS["blob512_iotf"]


@pytest.fixture(scope="module")
def pwf():
    from paper_2503_20146_gb300 import _build
    _build.build()
    from paper_2503_20146_gb300 import pwf as P
    P.load()
    return P


@pytest.mark.parametrize("batch,ny,nx,cluster", [(1, 128, 128, True), (64, 128, 128, False), (1, 64, 64, False),
                                                 (1, 256, 256, False), (4, 256, 256, False), (1, 512, 512, False),
                                                 (1, 128, 256, False)])
@pytest.mark.parametrize("coherent", [False, True])
def test_default_solver(pwf, batch, ny, nx, cluster, coherent):
    coh = 0.0 if coherent else W.xcoh_m

    def uses(flags):
        desc = pwf.PlanDesc(batch, ny, nx, W.pixel_m, W.wavelength_m, W.L1_m, W.L2_m, coh, coh, W.gamma, W.alpha.real,
                            W.alpha.imag, W.eta, flags | pwf.FLAG_NO_TUNE)
        with pwf.Plan(desc) as plan:
            return pwf.pwf_plan_uses_persistent(plan.handle)

    assert uses(0) == (2 if cluster else 0)
    if ny == nx:
        assert uses(pwf.FLAG_CLUSTER) == 2
