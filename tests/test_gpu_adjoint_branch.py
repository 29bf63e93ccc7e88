"""The branch of P_C that the reverse mode differentiates is the one that the update takes, at last-place ties too.

A uniform cell before its first update has a uniform z, which does not depend on gamma. gamma = sqrt(|z|^2) rounded
then ties in the last place: the update clips where |z|^2 exceeds gamma^2 as rounded, which sqrt(|z|^2) > gamma does not
show. With one update, d gamma_eff / d gamma is <z, A xi> / (|z| N) > 0 where it clips and 0 elsewhere."""

from fractions import Fraction

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2103_05968_gb300 import ccmf  # noqa: E402

DEV = "cuda:0"
SHAPE, BATCH, RHO = (2, 2, 2), 24, 0.7


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()


def rounded(x, bits):
    """A positive rational to `bits` significant bits, ties to even."""
    e = 0
    while x >= 2 ** bits:
        x, e = x / 2, e + 1
    while x < 2 ** (bits - 1):
        x, e = x * 2, e - 1
    return Fraction(round(x)) * Fraction(2) ** e


@pytest.mark.parametrize("precision", [ccmf.CCMF_FP64, ccmf.CCMF_FP32_MIXED])
def test_branch_at_last_place_ties(precision):
    f64 = precision == ccmf.CCMF_FP64
    dt, bits = (np.float64, 53) if f64 else (np.float32, 24)
    normals = np.random.default_rng(2).normal(size=(BATCH, 3))
    plan = ccmf.Plan(SHAPE, batch=BATCH, precision=precision, device=DEV)
    wide = torch.full((BATCH, *SHAPE), 10.0, dtype=plan.dtype, device=DEV)
    prm = ccmf.Params(fixed_iters=1, rho_rule=ccmf.CCMF_RHO_CONST, rho0=RHO)
    plan.solve(wide, normals, prm)
    z = plan.state()[1].cpu().numpy().reshape(BATCH, 6, -1)   # nothing clips: v = z
    assert (z == z[:, :, :1]).all()
    gamma, clips = np.empty(BATCH, dtype=dt), np.empty(BATCH, dtype=bool)
    for s in range(BATCH):
        n2 = Fraction(0)
        for c in z[s, :, 0]:
            n2 = rounded(Fraction(float(c)) ** 2 + n2, bits)
        gamma[s] = np.sqrt(dt(float(n2)))
        clips[s] = n2 > rounded(Fraction(float(gamma[s])) ** 2, bits)
    assert clips.any() and not clips.all()
    g = torch.from_numpy(gamma).to(DEV)[:, None, None, None].expand(BATCH, *SHAPE).contiguous()
    grad, _, _ = plan.gradient(g, normals, 1, 1, prm, rho_schedule=np.full((BATCH, 1), RHO))
    got = grad.cpu().numpy().reshape(BATCH, -1)
    plan.close()
    assert ((got > 0) == clips[:, None]).all()
    assert (got[~clips] == 0).all()
