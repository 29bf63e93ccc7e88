"""The reverse mode on plans tuned to other update variants: the same gradient as on the built-in one.

Every update of the reverse mode runs on k_update, whose rounding of a voxel does not depend on the variant, and the
penalties are given; the other passes are the same. What is left is the rounding of the forward run's FFT engines, none
here, so the bars (1e-10 of the largest entry in FP64, 1e-6 in FP32 arithmetic) only leave room for contraction."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from oracle import ccmf_adjoint as D  # noqa: E402
from paper_2103_05968_gb300 import ccmf  # noqa: E402
from paper_2103_05968_gb300 import microstructure as M  # noqa: E402

DEV = "cuda:0"
SHAPE, K, EVERY = (6, 8, 128), 12, 5
NORMAL = [0.36, 0.48, 0.8]


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()


def gradient(kind, gamma, sched):
    plan = ccmf.Plan(SHAPE, precision=ccmf.CCMF_FP64 if kind == "fp64" else ccmf.CCMF_FP32_MIXED, device=DEV)
    if kind == "mixed":
        plan.set_adjoint_forward(ccmf.CCMF_FP64)
    # a workspace that holds another call's values
    plan.workspace.fill_(63)
    grad, res, _ = plan.gradient(torch.from_numpy(gamma).to(DEV, plan.dtype), [NORMAL], K, EVERY, rho_schedule=sched)
    out = grad[0].double().cpu().numpy(), res[0]["gamma_eff"]
    plan.close()
    return out


@pytest.mark.parametrize("kind,bar", [("fp64", 1e-10), ("fp32", 1e-6), ("mixed", 1e-6)])
@pytest.mark.parametrize("variant", [0, 1, 3, 6, 9, 13])
def test_gradient_does_not_depend_on_the_update_variant(kind, bar, variant, monkeypatch):
    g = M.uniform_random(SHAPE, 0.5, 1.5, 11).astype(np.float32).astype(np.float64)
    sched = np.full((1, K), 0.9 * g.min())
    want, want_eff = gradient(kind, g, sched)
    monkeypatch.setenv("CCMF_UPDATE_VARIANT", str(variant))
    got, got_eff = gradient(kind, g, sched)
    assert np.abs(got - want).max() <= bar * np.abs(want).max()
    assert abs(got_eff - want_eff) <= bar * want_eff
    if kind == "fp64":
        J, ref = D.gradient(g, NORMAL, list(sched[0]))
        np.testing.assert_allclose(got, ref, rtol=0, atol=1e-9 * np.abs(ref).max())
        assert abs(got_eff - J) <= 1e-10 * J
