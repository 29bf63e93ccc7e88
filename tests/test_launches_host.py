"""Which kernels the entry points launch, on the stand-in CUDA runtime (CPU)."""

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
