"""The one-launch V-cycle on plans that differ in how planes and nodes are dealt:
several planes a CTA (8x8x32 in both precisions, 32x32x48, the largest level a
plan takes) and several nodes a thread (planes of 64 x 20), as the whole grid and
as the levels below a finest one.  The number of launches shows that the cycles
ran in one.  Oracle and tolerances as for the other plans: FP64 1e-12, FP32
16 x 2e-6 a refinement step."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle as O  # noqa: E402
from paper_1904_03808_gb300 import MG_MIXED, Context, binding, inputs as I  # noqa: E402

MU, K = I.TABLE1["mu"], I.TABLE1["K"]
LAM = I.lame_lambda(K, MU)


def rel(a, b):
    d = (a - b).ravel()
    return max(np.linalg.norm(d) / np.linalg.norm(b.ravel()), np.abs(d).max() / np.abs(b).max())


@pytest.mark.parametrize("shape", [(8, 8, 8), (8, 8, 32), (16, 8, 16)])
def test_fp64_vcycle_in_one_launch(shape):
    rng = np.random.default_rng(3)
    nx, ny, nz = shape
    b = I.rhs_field(5, nx, ny, nz)
    x = rng.uniform(-1, 1, (3, nz + 1, ny, nx))
    ctx = Context(nx, ny, nz, 2e-2 / nx, K, MU)
    bg, xg = torch.from_numpy(b).cuda(), torch.from_numpy(x.copy()).cuda()
    mg = O.MG(nx, ny, nz, LAM, MU)
    for _ in range(2):
        n0 = binding.launch_count()
        ctx.vcycle(bg, xg)
        assert binding.launch_count() - n0 == 1
        mg.vcycle(b, x)
    assert rel(xg.cpu().numpy(), x) <= 1e-12
    ctx.close()


# launches that a further cycle adds: none where the plan holds the whole grid;
# else four sweeps of two, two for the residual with its restriction, the plan
# and the prolongation
@pytest.mark.parametrize("shape,more", [((8, 8, 32), 0), ((32, 32, 48), 0), ((64, 20, 16), 0),
                                        ((128, 40, 32), 12)])
def test_fp32_inner_cycles_in_one_launch(shape, more):
    nx, ny, nz = shape
    b = I.rhs_field(6, nx, ny, nz)
    mg = O.MG(nx, ny, nz, LAM, MU)
    x, launches = np.zeros_like(b), []
    for cycles in (1, 2, 3):
        mg.vcycle(b, x)
        ctx = Context(nx, ny, nz, 2e-2 / nx, K, MU, precision=MG_MIXED, max_cycles=1,
                      inner_cycles=cycles)
        for _ in range(2):  # the second call starts from used buffers
            xg = torch.zeros(x.shape, dtype=torch.float64, device="cuda")
            n0 = binding.launch_count()
            ctx.solve(torch.from_numpy(b).cuda(), xg, tol=0.0)
            n = binding.launch_count() - n0
            assert rel(xg.cpu().numpy(), x) <= 3.2e-5
        launches.append(n)
        ctx.close()
    assert np.diff(launches).tolist() == [more, more]
