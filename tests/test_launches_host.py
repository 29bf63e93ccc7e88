"""Which kernels the entry points launch, on the stand-in CUDA runtime (CPU)."""

import re

import pytest

from fake_cuda import needs_toolchain, run_fake

pytestmark = needs_toolchain

_PLAN = """
def plan_for(shape, batch, precision, **knobs):
    code, h = ccmf.ccmf_plan_create(*shape, batch, precision)
    assert code == 0
    if knobs:
        assert ccmf.ccmf_plan_set_tuning(h, knobs) == 0, knobs
    return h, ccmf.ccmf_plan_workspace_bytes(h)[1]
"""


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2103_05968_gb300 import _build
    _build.build()


@pytest.mark.parametrize("precision", ["fp64", "fp32", "mixed"])
@pytest.mark.parametrize("variant", [0, 1, 3, 7, 9, 11, 12, 13])
def test_gradient_runs_its_updates_on_the_kernel_that_writes_z(variant, precision, tmp_path):
    """The reverse sweep reads z = v + rho xi of every update, which only k_update writes, whatever update variant the
    plan, or the FP64 plan behind an FP32 one, is tuned to."""
    body = _PLAN + f"""
prec = ccmf.CCMF_FP64 if {precision!r} == "fp64" else ccmf.CCMF_FP32_MIXED
shape, K, every = (6, 8, 128), 4, 2
h, n = plan_for(shape, 1, prec)
if {precision!r} == "mixed":
    assert ccmf.ccmf_set_adjoint_forward(h, ccmf.CCMF_FP64) == 0
ws, an = buf(n), ccmf.ccmf_adjoint_workspace_bytes(h, K, every)[1]
launches()
N = 6 * 8 * 128
code = ccmf.ccmf_adjoint(h, buf(8 * N), 0, [0.0, 0.6, 0.8], ccmf.Params().to_c(), K, every, np.full((1, K), 0.5), ws, n,
                         buf(an), an, buf(8 * N), np.zeros((1, K)), None, None)
assert code == 0, code
out["kernels"] = [k for _, k, _, _ in launches()]
"""
    kernels = run_fake(body, tmp_path, env={"CCMF_UPDATE_VARIANT": str(variant)})["kernels"]
    updates = [k for k in kernels if "k_update" in k]
    # 4 replayed, 1 final evaluation, 4 recomputed, and the final evaluation of each of 4 reverse steps
    assert len(updates) == 13
    assert all("8k_updateI" in k for k in updates), sorted(set(updates))


# kernels that load gamma in vectors: k_update on 2 or 4 voxels, the TMA and stored-divergence updates
_VECTOR = r"8k_updateI[fd]Li[24]E|k_update_(pipe|tma|ab|abw)I"


def _vector_kernels(names):
    return sorted({k for k in names if re.search(_VECTOR, k)})


@pytest.mark.parametrize("double", [False, True])
@pytest.mark.parametrize("variant", [None, 0, 3, 9, 13])
@pytest.mark.parametrize("call", ["solve", "adjoint"])
def test_odd_gamma_stride_takes_scalar_loads(call, variant, double, tmp_path):
    """Field s of a batch starts at gamma + s stride: with an odd stride every second field is off the alignment of a
    pair, though the base address and N3 are even."""
    body = _PLAN + f"""
N = 6 * 8 * 128
K = 2
prm = ccmf.Params(fixed_iters=K).to_c()
def names(batch, stride):
    h, n = plan_for((6, 8, 128), batch, ccmf.CCMF_FP64 if {double} else ccmf.CCMF_FP32_MIXED)
    an = ccmf.ccmf_adjoint_workspace_bytes(h, K, K)[1]
    xi = [[0.0, 0.6, 0.8]] * batch
    launches()
    if {call!r} == "solve":
        code = ccmf.ccmf_solve(h, buf(8 * batch * (N + 1)), stride, xi, prm, buf(n), n, None, None, None, None)
    else:
        code = ccmf.ccmf_adjoint(h, buf(8 * batch * (N + 1)), stride, xi, prm, K, K, np.full((batch, K), 0.5), buf(n),
                                 n, buf(an), an, buf(8 * batch * N), None, None, None)
    assert code == 0, code
    return [k for _, k, _, _ in launches()]
out["one"], out["even"], out["odd"] = names(1, N + 1), names(2, N), names(2, N + 1)
"""
    got = run_fake(body, tmp_path, env={} if variant is None else {"CCMF_UPDATE_VARIANT": str(variant)})
    assert _vector_kernels(got["odd"]) == []
    assert got["one"] and got["even"]
    assert _vector_kernels(got["even"]) == _vector_kernels(got["one"]) != []


@pytest.mark.parametrize("double", [False, True])
@pytest.mark.parametrize("persistent", [False, True])
@pytest.mark.parametrize("variant", [None, 0, 3, 9, 13])
def test_batch_with_an_unaligned_gamma_takes_scalar_loads(variant, persistent, double, tmp_path):
    body = f"""
N = 6 * 8 * 128
es = 8 if {double} else 4
code, h = ccmf.ccmf_batch_create([(6, 8, 128)] * 2, ccmf.CCMF_FP64 if {double} else ccmf.CCMF_FP32_MIXED)
assert code == 0
assert ccmf.ccmf_batch_set_persistent(h, {int(persistent)}) == 0
n = ccmf.ccmf_batch_workspace_bytes(h)[1]
def names(offset):
    launches()
    g = [buf(8 * N).value, buf(8 * N, offset).value]
    ws = buf(n)
    code = ccmf.ccmf_batch_solve(h, g, [[0, 0.6, 0.8]] * 2, ccmf.Params(fixed_iters=2).to_c(), ws, n, None, None)
    assert code == 0, code
    k = [k for _, k, _, _ in launches()]
    # the timing runs of the tuning take every update variant over the same fields
    code, _ = ccmf.ccmf_batch_autotune(h, g, [[0, 0.6, 0.8]] * 2, ws, n, 2, 1, None)
    assert code == 0, code
    return k, [k for _, k, _, _ in launches()]
out["unaligned"], out["tuned"] = names(es)
"""
    got = run_fake(body, tmp_path, env={} if variant is None else {"CCMF_UPDATE_VARIANT": str(variant)})
    assert got["unaligned"] and got["tuned"]
    assert _vector_kernels(got["unaligned"]) == []
    assert _vector_kernels(got["tuned"]) == []


def test_state_export_runs_on_the_device_of_its_plan(tmp_path):
    """Exporting a compact FP32 state launches a kernel: on the plan's device, whichever is current, and the caller's
    current device stays."""
    body = _PLAN + """
h, n = plan_for((6, 8, 16), 1, ccmf.CCMF_FP32_MIXED)
N = 6 * 8 * 16
ws, e, v = buf(n), buf(24 * N), buf(24 * N)
assert ccmf.ccmf_state_import(h, ws, e, v, [0.5], [12345], None) == 0
words = np.ctypeslib.as_array(ctypes.cast(ws, ctypes.POINTER(ctypes.c_int32)), (64,))   # the scalars of solve 0
assert (words == 12345).sum() == 1
imported = words.copy()
launches()
set_device(3)
seen = []
# which word holds the mark of a compact state is the library's own business: try them all
for i in range(64):
    for mark in (12345, 12346):
        words[:] = imported
        if words[i] == 12345:
            continue
        words[i] = mark
        code, rho, iters = ccmf.ccmf_state_export(h, ws, e, v, 1, None)
        assert code == 0
        seen += [(d, k) for d, k, _, _ in launches()]
out["seen"] = seen
d = ctypes.c_int()
fake.cudaGetDevice(ctypes.byref(d))
out["current"] = d.value
"""
    got = run_fake(body, tmp_path)
    assert len(got["seen"]) == 1 and "k_state_to_ev" in got["seen"][0][1]
    assert got["seen"][0][0] == 0
    assert got["current"] == 3


def test_cleared_workspace_holds_no_compact_state(tmp_path):
    """Zeroed memory exports as it is: nothing in it reads as a compact state, whose expansion divides by the penalty."""
    body = _PLAN + """
h, n = plan_for((6, 8, 16), 2, ccmf.CCMF_FP32_MIXED)
N = 6 * 8 * 16
e, v = (np.ones(12 * N, dtype=np.float32) for _ in range(2))
launches()
code, rho, iters = ccmf.ccmf_state_export(h, buf(n), ctypes.c_void_p(e.ctypes.data), ctypes.c_void_p(v.ctypes.data), 2,
                                          None)
out["code"], out["launches"] = code, launches()
out["values"] = [float(np.abs(e).max()), float(np.abs(v).max()), float(max(rho)), int(max(iters))]
"""
    got = run_fake(body, tmp_path)
    assert got == {"code": 0, "launches": [], "values": [0.0, 0.0, 0.0, 0]}


def test_plane_pass_by_environment(tmp_path):
    """CCMF_PLANE_FUSED: 0 the line passes, another value the plane pass where a plane fits a block, unset the
    built-in rule (in FP64 the line passes unless the planes fill the SMs twice)."""
    body = _PLAN + """
def info(shape, double):
    h, _ = plan_for(shape, 1, ccmf.CCMF_FP64 if double else ccmf.CCMF_FP32_MIXED)
    return ccmf.ccmf_plan_launch_info(h)[1]["plane_blocks"]
out["fused"] = [info((80, 80, 80), True), info((80, 80, 80), False), info((512, 512, 16), True)]
"""
    assert run_fake(body, tmp_path)["fused"] == [0, 1, 0]
    assert run_fake(body, tmp_path, env={"CCMF_PLANE_FUSED": "1"})["fused"] == [1, 1, 0]
    assert run_fake(body, tmp_path, env={"CCMF_PLANE_FUSED": "0"})["fused"] == [0, 0, 0]


@pytest.mark.parametrize("double", [False, True])
@pytest.mark.parametrize("variant", [0, 11, 12])
@pytest.mark.parametrize("shape,batch", [((6, 8, 16), 1), ((64, 64, 64), 3), ((128, 128, 128), 1), ((50, 48, 32), 7)])
def test_launch_info_names_the_grid_of_the_update_pass(shape, batch, variant, double, tmp_path):
    body = _PLAN + f"""
shape, batch = {shape}, {batch}
h, n = plan_for(shape, batch, ccmf.CCMF_FP64 if {double} else ccmf.CCMF_FP32_MIXED, update_variant={variant})
N = shape[0] * shape[1] * shape[2]
launches()
code = ccmf.ccmf_solve(h, buf(8 * N), 0, [[0, 0.6, 0.8]] * batch, ccmf.Params(fixed_iters=2).to_c(), buf(n), n, None, None,
                       None, None)
assert code == 0
out["grids"] = [g for _, k, g, _ in launches() if "k_update" in k][:-1]    # the last is the final evaluation
out["said"] = ccmf.ccmf_plan_launch_info(h)[1]["update_blocks"]
"""
    got = run_fake(body, tmp_path)
    # the smallest grid is that of the branch with the most solves
    assert min(got["grids"]) == got["said"]
