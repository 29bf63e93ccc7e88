"""The register update pass on the compact FP32 state (z and the projection factor s in place of e and v), the pair
and strided thread groups, the plane pass and the chunk rules, at the sizes where they can go wrong.

One step from an exported state against the FP64 oracle: the bars of test_gpu_fp32_parity (the FP32 step rounds w, d,
the FFT pair and the projection to a few eps32 log2 N of the largest term; P_C is 1-Lipschitz), 1e-5 of the largest
of max|e|, max|v|. Two engines of the FP64 Poisson solve differ by rounding alone, a few eps64 log2 N per update;
three updates and the factor 2 per update of the relaxed step leave them within 1e-12 of the largest value."""

import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from oracle import ccmf_oracle as O  # noqa: E402
from paper_2103_05968_gb300 import ccmf  # noqa: E402
from paper_2103_05968_gb300 import microstructure as M  # noqa: E402

DEV = "cuda:0"
FIELD_REL = 1e-5
NORMAL = [0.36, 0.48, 0.8]


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()


def field(shape, dtype, offset=0):
    """Random field on the GPU whose first element lies `offset` elements past an aligned address."""
    g = M.uniform_random(shape, 0.4, 1.5, 7).astype(dtype)
    buf = torch.empty(g.size + offset, dtype=torch.from_numpy(g).dtype, device=DEV)
    view = buf[offset:].view(shape)
    view.copy_(torch.from_numpy(g))
    return g.astype(np.float64), view


# single axes, odd N3 (strided pairs), N3 = 2 mod 4 (pairs), a partial last chunk, gamma off the vector alignment;
# variant None: the built-in one
@pytest.mark.parametrize("shape,offset,variant", [
    ((1, 1, 20), 0, 12), ((9, 5, 1), 0, None), ((5, 6, 3), 0, None), ((6, 10, 15), 0, None), ((3, 4, 2), 0, None),
    ((8, 12, 18), 0, None), ((8, 8, 9), 0, None), ((30, 32, 16), 1, 12), ((30, 32, 16), 0, 11), ((30, 32, 16), 2, 11),
    ((30, 32, 16), 0, 0), ((30, 32, 16), 2, 0), ((12, 10, 30), 2, None), ((64, 8, 10), 3, None)])
def test_one_step_on_the_compact_state(shape, offset, variant):
    g64, g = field(shape, np.float32, offset)
    plan = ccmf.Plan(shape, precision=ccmf.CCMF_FP32_MIXED, device=DEV)
    if variant is not None:
        plan.set_tuning(update_variant=variant)
    plan.solve(g, [NORMAL], ccmf.Params(fixed_iters=6))
    e0, v0, rho0, _ = plan.state()
    plan.solve(g, [NORMAL], ccmf.Params(fixed_iters=1, resume=1))
    e1, v1, rho1, it1 = plan.state()
    plan.close()
    assert it1[0] == 7
    e0s, v0s = (x[0].cpu().numpy().astype(np.float64) for x in (e0, v0))
    xi = np.asarray(NORMAL) / np.linalg.norm(NORMAL)
    _, e_ref, v_ref = O.admm_step(e0s, v0s, rho0[0], g64, xi, 0.25)
    scale = max(np.abs(e_ref).max(), np.abs(v_ref).max())
    assert np.abs(e1[0].cpu().numpy() - e_ref).max() <= FIELD_REL * scale
    assert np.abs(v1[0].cpu().numpy() - v_ref).max() <= FIELD_REL * scale
    assert abs(rho1[0] - O.next_rho(rho0[0], O.RHO_BB, e0s, e_ref, v0s, v_ref, O.Params())) <= 1e-4 * rho1[0]


@pytest.mark.parametrize("shape", [(16, 16, 16), (6, 10, 15), (8, 12, 18)])
def test_exported_state_continues_bit_for_bit(shape):
    _, g = field(shape, np.float32)
    plan = ccmf.Plan(shape, precision=ccmf.CCMF_FP32_MIXED, device=DEV)
    plan.solve(g, [NORMAL], ccmf.Params(fixed_iters=6))
    saved = plan.state()
    plan.solve(g, [NORMAL], ccmf.Params(fixed_iters=4, resume=1))
    want = plan.state()
    fresh = ccmf.Plan(shape, precision=ccmf.CCMF_FP32_MIXED, device=DEV)
    fresh.load_state(*saved)
    fresh.solve(g, [NORMAL], ccmf.Params(fixed_iters=4, resume=1))
    got = fresh.state()
    assert torch.equal(want[0], got[0]) and torch.equal(want[1], got[1])
    assert list(want[2]) == list(got[2]) and list(want[3]) == list(got[3])
    plan.close()
    fresh.close()


# one step after the update pass changes between variants that keep (z, s) and (e, v)
@pytest.mark.parametrize("first,then", [(12, 11), (12, 3), (3, 12), (0, 7), (12, 9), (9, 12)])
def test_update_variant_changes_between_state_formats(first, then):
    shape = (6, 8, 128)
    _, g = field(shape, np.float32)
    out = []
    for second in (first, then):
        plan = ccmf.Plan(shape, precision=ccmf.CCMF_FP32_MIXED, device=DEV)
        plan.set_tuning(update_variant=first)
        plan.solve(g, [NORMAL], ccmf.Params(fixed_iters=6))
        if second != first:
            plan.set_tuning(update_variant=second)
        plan.solve(g, [NORMAL], ccmf.Params(fixed_iters=1, resume=1))
        e, v, rho, it = plan.state()
        out.append((e.cpu().numpy(), v.cpu().numpy(), rho[0], it[0]))
        plan.close()
    (e, v, rho, it), (e2, v2, rho2, it2) = out
    scale = max(np.abs(e).max(), np.abs(v).max())
    assert it == it2 == 7
    assert np.abs(e - e2).max() <= FIELD_REL * scale and np.abs(v - v2).max() <= FIELD_REL * scale
    assert abs(rho - rho2) <= 1e-4 * rho


# axes of one element, of one stage and of several, odd pitches, the two launch sizes (more planes than SMs)
@pytest.mark.parametrize("shape,batch", [((1, 12, 6), 1), ((12, 1, 6), 1), ((2, 3, 10), 1), ((8, 2, 10), 2),
                                         ((25, 27, 4), 1), ((100, 90, 4), 1), ((80, 75, 6), 1), ((16, 16, 30), 20)])
@pytest.mark.parametrize("precision", [ccmf.CCMF_FP64, ccmf.CCMF_FP32_MIXED])
def test_plane_pass_against_line_passes(shape, batch, precision):
    f64 = precision == ccmf.CCMF_FP64
    _, g = field(shape, np.float64 if f64 else np.float32)
    normals = np.random.default_rng(3).normal(size=(batch, 3))
    out = []
    for planes in (1, 0):
        plan = ccmf.Plan(shape, batch=batch, precision=precision, device=DEV)
        plan.set_tuning(plane_blocks=planes)
        plan.solve(g, normals, ccmf.Params(fixed_iters=3 if f64 else 1))
        out.append([x.cpu().numpy() for x in plan.state()[:2]])
        plan.close()
    scale = max(np.abs(x).max() for x in out[1])
    for a, b in zip(*out):
        assert np.abs(a - b).max() <= (1e-12 if f64 else FIELD_REL) * scale


def test_allocation_free_solve_with_more_chunks_than_blocks():
    """64 x 64 x 60 in FP64: 960 chunks of partial sums, more than the scratch area's block slots."""
    shape = (64, 64, 60)
    _, g = field(shape, np.float64)
    plan = ccmf.Plan(shape, precision=ccmf.CCMF_FP64, device=DEV)
    want, _, _ = plan.solve(g, [NORMAL], ccmf.Params(fixed_iters=10))
    plan.close()
    res = ccmf.ccmf_result()
    prm = ccmf.Params(fixed_iters=10).to_c()
    code = ccmf.ccmf_solve_static(*shape, ccmf.CCMF_FP64, ctypes.c_void_p(g.data_ptr()), NORMAL, prm, None, None,
                                  ctypes.byref(res), ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    torch.cuda.synchronize()
    assert code == ccmf.CCMF_OK
    assert abs(res.gamma_eff - want[0]["gamma_eff"]) <= 1e-12 * abs(res.gamma_eff)
    assert abs(res.residual - want[0]["residual"]) <= 1e-9 * res.residual
