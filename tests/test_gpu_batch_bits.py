"""A solve of a batch is its solo solve bit for bit, though the launch shapes (lines per block, the FP64 plane pass, its
block size) follow the number of solves: fields, penalties and reported numbers after a few adaptive updates."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2103_05968_gb300 import ccmf  # noqa: E402
from paper_2103_05968_gb300 import microstructure as M  # noqa: E402

DEV = "cuda:0"


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()


# batches whose planes fill the SMs twice (FP64 takes the plane pass there and the line passes alone), odd axes, every
# radix, an axis with warp lines, N3 with the warp z passes
@pytest.mark.parametrize("shape,batch", [((16, 16, 16), 34), ((24, 20, 16), 34), ((27, 25, 10), 52), ((10, 9, 15), 40),
                                         ((1, 12, 6), 80), ((128, 10, 6), 80), ((6, 10, 128), 5), ((32, 32, 32), 3)])
@pytest.mark.parametrize("precision", [ccmf.CCMF_FP64, ccmf.CCMF_FP32_MIXED])
def test_batch_solve_is_its_solo_solve(shape, batch, precision):
    g = M.random_two_phase(shape, 0.3, 0.25, 1.0, 7)
    dt = torch.float64 if precision == ccmf.CCMF_FP64 else torch.float32
    gt = torch.from_numpy(g).to(DEV, dt)
    normals = np.random.default_rng(3).normal(size=(batch, 3))
    prm = ccmf.Params(fixed_iters=6)
    plan = ccmf.Plan(shape, batch=batch, precision=precision, device=DEV)
    res, flow, cut = plan.solve(gt, normals, prm, want_flow=True, want_cut=True)
    plan.close()
    solo = ccmf.Plan(shape, precision=precision, device=DEV)
    for s in (0, batch // 2, batch - 1):
        r, f, c = solo.solve(gt, normals[s:s + 1], prm, want_flow=True, want_cut=True)
        assert torch.equal(f[0], flow[s]) and torch.equal(c[0], cut[s])
        assert r[0] == res[s]
    solo.close()
