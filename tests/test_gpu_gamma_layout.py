"""Gamma fields off the alignment of the vector loads: padded fields of a batch with an odd stride.

With a constant penalty no sum enters the state, and the rounding of a voxel does not depend on the thread group that
processes it, so the fields are those of the contiguous layout bit for bit. In the reverse mode the forward passes are
the same too; its sums are taken voxel by voxel."""

import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2103_05968_gb300 import ccmf  # noqa: E402
from paper_2103_05968_gb300 import microstructure as M  # noqa: E402

DEV = "cuda:0"
NORMALS = [[0.36, 0.48, 0.8], [0.6, 0.0, 0.8]]


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()


def padded(fields, stride):
    n = fields[0].numel()
    buf = torch.zeros(stride * len(fields), dtype=fields[0].dtype, device=DEV)
    for s, f in enumerate(fields):
        buf[s * stride:s * stride + n] = f.flatten()
    return buf


@pytest.mark.parametrize("precision", [ccmf.CCMF_FP64, ccmf.CCMF_FP32_MIXED])
@pytest.mark.parametrize("shape,variant", [((6, 5, 10), None), ((8, 6, 12), None), ((8, 6, 12), 0), ((6, 8, 128), 3),
                                           ((6, 8, 128), 9), ((6, 8, 128), 13)])
def test_padded_batch_with_an_odd_stride(shape, variant, precision):
    n = int(np.prod(shape))
    dt = torch.float64 if precision == ccmf.CCMF_FP64 else torch.float32
    fields = [torch.from_numpy(M.uniform_random(shape, 0.5, 1.5, s)).to(DEV, dt) for s in (3, 4)]
    prm = ccmf.Params(fixed_iters=5, rho_rule=ccmf.CCMF_RHO_CONST, rho0=0.4)
    out = []
    for stride in (n, n + 1):
        plan = ccmf.Plan(shape, batch=2, precision=precision, device=DEV)
        if variant is not None and stride == n + 1:
            plan.set_tuning(update_variant=variant)
        g = padded(fields, stride)
        cut = torch.empty((2, 6, *shape), dtype=dt, device=DEV)
        flow = torch.empty((2, 3, *shape), dtype=dt, device=DEV)
        code = ccmf.ccmf_solve(plan.handle, ctypes.c_void_p(g.data_ptr()), stride, NORMALS, prm.to_c(),
                               ctypes.c_void_p(plan.ws_ptr), plan.workspace_bytes, ctypes.c_void_p(flow.data_ptr()),
                               ctypes.c_void_p(cut.data_ptr()), None,
                               ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
        assert code == ccmf.CCMF_OK
        abytes = ccmf.ccmf_adjoint_workspace_bytes(plan.handle, 4, 2)[1]
        aws = torch.empty(abytes + 256, dtype=torch.uint8, device=DEV)
        grad = torch.empty((2, *shape), dtype=dt, device=DEV)
        code = ccmf.ccmf_adjoint(plan.handle, ctypes.c_void_p(g.data_ptr()), stride, NORMALS, prm.to_c(), 4, 2,
                                 np.full((2, 4), 0.4), ctypes.c_void_p(plan.ws_ptr), plan.workspace_bytes,
                                 ctypes.c_void_p((aws.data_ptr() + 255) // 256 * 256), abytes,
                                 ctypes.c_void_p(grad.data_ptr()), None, None,
                                 ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
        assert code == ccmf.CCMF_OK
        torch.cuda.synchronize()
        out.append((flow, cut, grad))
        plan.close()
    for want, got in zip(*out):
        assert torch.isfinite(want).all()
        assert torch.equal(want, got)


# The fields are the same bits again; the reported numbers are sums in another grouping, a few eps of each sum: 1e-5 in
# FP32, 1e-12 in FP64. (The residual is a mean of squares of differences; it is compared at the same bar of |<v>|.)
@pytest.mark.parametrize("precision,bar", [(ccmf.CCMF_FP64, 1e-12), (ccmf.CCMF_FP32_MIXED, 1e-5)])
@pytest.mark.parametrize("variant", [None, 3, 9, 13])
def test_batch_with_an_unaligned_gamma(variant, precision, bar, monkeypatch):
    if variant is not None:
        monkeypatch.setenv("CCMF_UPDATE_VARIANT", str(variant))
    dt = torch.float64 if precision == ccmf.CCMF_FP64 else torch.float32
    shapes = [(6, 8, 128), (6, 8, 128), (5, 9, 15), (6, 5, 10)]
    fields = [torch.from_numpy(M.uniform_random(sh, 0.5, 1.5, s)).to(DEV, dt) for s, sh in enumerate(shapes)]
    normals = np.array([NORMALS[0], NORMALS[1], NORMALS[0], NORMALS[1]])
    prm = ccmf.Params(fixed_iters=5, rho_rule=ccmf.CCMF_RHO_CONST, rho0=0.4)
    out = []
    for offset, persistent in ((0, False), (1, False), (0, True), (1, True)):
        gammas = []
        for f in fields:
            buf = torch.zeros(f.numel() + offset, dtype=dt, device=DEV)
            buf[offset:] = f.flatten()
            gammas.append(buf[offset:])
        batch = ccmf.Batch(shapes, precision=precision, device=DEV)
        batch.set_persistent(persistent)
        out.append(batch.solve(gammas, normals, prm))
        batch.close()
    for other in out[1:]:
        for a, b in zip(out[0], other):
            assert a["status"] == b["status"] == 0 and a["iters"] == b["iters"]
            assert abs(a["gamma_eff"] - b["gamma_eff"]) <= bar * abs(a["gamma_eff"])
            assert abs(a["gamma_primal"] - b["gamma_primal"]) <= bar * abs(a["gamma_primal"])
            assert abs(a["residual"] - b["residual"]) <= bar * a["mean_v_norm"]
