"""The branch of P_C that the reverse mode differentiates is the one that the update takes, at last-place ties too.

A uniform cell before its first update has a uniform z, which does not depend on gamma. gamma = sqrt(|z|^2) rounded
then ties in the last place, and its predecessor lies one place below. The FP64 update clips where the rounded root
exceeds gamma, the FP32 update where |z|^2 exceeds gamma^2 as rounded. With one update, d gamma_eff / d gamma is
<z, A xi> / (|z| N) > 0 where it clips and 0 elsewhere.

The same tie is every default start: rho0 = min gamma, |A xi| = 1, so |z| = min gamma up to rounding on the weakest
phase, and nothing clips. The LTD rule keeps rho as long as e' = 0; an update that takes the rounding error of |z|^2 for
a clipped voxel sends it to its bound."""

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


def norm2(z, bits):
    """|z|^2 by the chain of fused operations in which the passes add it."""
    n2 = Fraction(0)
    for c in z:
        n2 = rounded(Fraction(float(c)) ** 2 + n2, bits) if c else n2
    return n2


@pytest.mark.parametrize("precision", [ccmf.CCMF_FP64, ccmf.CCMF_FP32_MIXED])
def test_branch_at_last_place_ties(precision):
    f64 = precision == ccmf.CCMF_FP64
    dt, bits = (np.float64, 53) if f64 else (np.float32, 24)
    normals = np.tile(np.random.default_rng(2).normal(size=(BATCH // 2, 3)), (2, 1))
    plan = ccmf.Plan(SHAPE, batch=BATCH, precision=precision, device=DEV)
    wide = torch.full((BATCH, *SHAPE), 10.0, dtype=plan.dtype, device=DEV)
    prm = ccmf.Params(fixed_iters=1, rho_rule=ccmf.CCMF_RHO_CONST, rho0=RHO)
    plan.solve(wide, normals, prm)
    z = plan.state()[1].cpu().numpy().reshape(BATCH, 6, -1)   # nothing clips: v = z
    assert (z == z[:, :, :1]).all()
    gamma, clips = np.empty(BATCH, dtype=dt), np.empty(BATCH, dtype=bool)
    for s in range(BATCH):
        n2 = norm2(z[s, :, 0], bits)
        root = np.sqrt(dt(float(n2)))
        gamma[s] = root if s < BATCH // 2 else np.nextafter(root, dt(0))
        clips[s] = root > gamma[s] if f64 else n2 > rounded(Fraction(float(gamma[s])) ** 2, bits)
    assert clips.any() and not clips.all()
    g = torch.from_numpy(gamma).to(DEV)[:, None, None, None].expand(BATCH, *SHAPE).contiguous()
    grad, _, _ = plan.gradient(g, normals, 1, 1, prm, rho_schedule=np.full((BATCH, 1), RHO))
    got = grad.cpu().numpy().reshape(BATCH, -1)
    plan.close()
    assert ((got > 0) == clips[:, None]).all()
    assert (got[~clips] == 0).all()


def test_default_start_of_the_ltd_rule_in_fp64():
    batch, shape, low = 64, (4, 3, 2), 0.3
    normals = np.random.default_rng(6).normal(size=(batch, 3))
    plan = ccmf.Plan(shape, batch=batch, precision=ccmf.CCMF_FP64, device=DEV)
    plan.solve(torch.full(shape, 10.0, dtype=plan.dtype, device=DEV), normals,
               ccmf.Params(fixed_iters=1, rho_rule=ccmf.CCMF_RHO_CONST, rho0=low))
    z = plan.state()[1].cpu().numpy().reshape(batch, 6, -1)
    assert (z == z[:, :, :1]).all()
    two = torch.full(shape, 1.0, dtype=plan.dtype, device=DEV)
    two[:2] = low
    res, _, _ = plan.solve(two, normals, ccmf.Params(fixed_iters=1, rho_rule=ccmf.CCMF_RHO_LTD))
    e = plan.state()[0].cpu().numpy().reshape(batch, -1)
    plan.close()
    below = np.array([np.sqrt(float(norm2(z[s, :, 0], 53))) <= low for s in range(batch)])
    assert below.sum() >= batch // 2
    assert (e[below] == 0).all()
    assert all(res[s]["rho"] == low for s in range(batch) if below[s])


@pytest.mark.parametrize("low", [0.1, 0.25, 0.3, 0.37, 0.45, 1.0])
@pytest.mark.parametrize("delta", [0.25, 0.5])
def test_ltd_rule_keeps_the_default_penalty(low, delta):
    """The first update of the default start clips nothing in exact arithmetic. An emulation of its roundings on 3000
    random normals (exact rationals) keeps rho for 92 % and more of them at every case here, and for axis normals; 85 %
    of 300 leaves four standard deviations."""
    batch, shape = 303, (4, 3, 2)
    normals = np.concatenate([np.eye(3), np.random.default_rng(8).normal(size=(batch - 3, 3))])
    plan = ccmf.Plan(shape, batch=batch, precision=ccmf.CCMF_FP64, device=DEV)
    two = torch.full(shape, 2.0, dtype=plan.dtype, device=DEV)
    two[:2] = low
    res, _, _ = plan.solve(two, normals, ccmf.Params(fixed_iters=1, rho_rule=ccmf.CCMF_RHO_LTD, delta=delta))
    plan.close()
    kept = np.array([r["rho"] == low for r in res])
    assert kept[:3].all()
    assert kept[3:].mean() >= 0.85
