"""The FP64 projection over the range of its operands.

Within 2^-100 <= |z|^2 < 2^100 the scale of P_C and the norm come from a Halley step on the FP32 reciprocal square root,
outside from the library's square root and division. Scaling gamma and a constant penalty by a power of two scales v and
the reported energies by it and leaves e as it is, exactly in every other operation, so the two forms meet in one
comparison; where they differ it is by a few eps64 per update. Five updates of the relaxed step at most double an error
each: 1e-13 of the largest value. gamma = 0 (pores) and cells on both sides of the switch are among the voxels."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2103_05968_gb300 import ccmf  # noqa: E402

DEV = "cuda:0"
SHAPE = (12, 10, 8)
NORMAL = [0.36, 0.48, 0.8]


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()


def run(power, variant):
    rng = np.random.default_rng(4)
    g = rng.uniform(0.25, 4.0, SHAPE)
    g[rng.random(SHAPE) < 0.2] = 0.0
    plan = ccmf.Plan(SHAPE, precision=ccmf.CCMF_FP64, device=DEV)
    plan.set_tuning(update_variant=variant)
    scale = 2.0 ** power
    res, _, cut = plan.solve(torch.from_numpy(g * scale).to(DEV), [NORMAL],
                             ccmf.Params(fixed_iters=5, rho_rule=ccmf.CCMF_RHO_CONST, rho0=0.5 * scale), want_cut=True)
    e, v, _, _ = plan.state()
    plan.close()
    assert res[0]["status"] == 0
    return (e.cpu().numpy(), v.cpu().numpy() / scale, cut.cpu().numpy(),
            np.array([res[0]["gamma_eff"] / scale, res[0]["gamma_primal"] / scale, res[0]["residual"]]))


@pytest.mark.parametrize("variant", [0, 11])
@pytest.mark.parametrize("power", [-300, -120, -51, -50, -49, 49, 50, 51, 120, 300])
def test_scaled_cell_gives_the_scaled_solution(power, variant):
    for want, got in zip(run(0, variant), run(power, variant)):
        assert np.isfinite(got).all()
        assert np.abs(got - want).max() <= 1e-13 * np.abs(want).max()
