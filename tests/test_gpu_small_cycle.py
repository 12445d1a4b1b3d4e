"""The one-launch V-cycle of the small levels (one 16-CTA cluster holding
every level in shared memory) against the oracle's V-cycles, in FP64 through
mg_vcycle and in FP32 through one refinement step of the mixed solve with a
fixed number of inner cycles.

Shapes: one plane a CTA and fewer (8, 16 planes), several (33 and more), nx !=
ny, an odd coarsest level (80 x 40 x 40 -> 10 x 5 x 5), planes that only fit
one at a time (48 x 48 x 24: three interior planes a CTA do not fit twice),
grids on which the kernel starts at level 1, and unequal sweep counts
including none.

Tolerances: FP64 1e-12 as everywhere.  FP32: a pair of sweeps is held to 2e-6
(30 units of rounding); a V-cycle has two pairs and three transfers on each of
about four levels, and the cycles of one refinement step contract earlier
errors, so 16 x 2e-6 = 3.2e-5 relative to the step's correction."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle as O  # noqa: E402
from paper_1904_03808_gb300 import MG_MIXED, Context, inputs as I  # noqa: E402

MU, K = I.TABLE1["mu"], I.TABLE1["K"]
LAM = I.lame_lambda(K, MU)

SHAPES = [(8, 8, 8), (16, 8, 12), (32, 16, 16), (24, 40, 20), (64, 16, 32), (40, 40, 40),
          (48, 48, 24), (80, 40, 40), (64, 64, 64)]
SWEEPS = [(2, 2), (1, 3), (0, 2), (1, 0)]


def rel(a, b):
    d = (a - b).ravel()
    return max(np.linalg.norm(d) / np.linalg.norm(b.ravel()), np.abs(d).max() / np.abs(b).max())


def _cases():
    return [(s, (2, 2)) for s in SHAPES] + [((32, 32, 32), n) for n in SWEEPS[1:]]


@pytest.mark.parametrize("shape,nu", _cases())
def test_fp64_vcycle(shape, nu):
    rng = np.random.default_rng(3)
    nx, ny, nz = shape
    b = I.rhs_field(5, nx, ny, nz)
    x = rng.uniform(-1, 1, (3, nz + 1, ny, nx))  # walls included
    ctx = Context(nx, ny, nz, 2e-2 / nx, K, MU, nu1=nu[0], nu2=nu[1])
    bg, xg = torch.from_numpy(b).cuda(), torch.from_numpy(x.copy()).cuda()
    mg = O.MG(nx, ny, nz, LAM, MU, *nu)
    for _ in range(2):
        ctx.vcycle(bg, xg)
        mg.vcycle(b, x)
    assert rel(xg.cpu().numpy(), x) <= 1e-12
    ctx.close()


@pytest.mark.parametrize("shape,nu", _cases())
@pytest.mark.parametrize("cycles", [1, 3])
def test_fp32_inner_cycles(shape, nu, cycles):
    nx, ny, nz = shape
    b = I.rhs_field(6, nx, ny, nz)
    x = np.zeros_like(b)
    ctx = Context(nx, ny, nz, 2e-2 / nx, K, MU, precision=MG_MIXED, nu1=nu[0], nu2=nu[1],
                  max_cycles=1, inner_cycles=cycles)
    mg = O.MG(nx, ny, nz, LAM, MU, *nu)
    for _ in range(cycles):
        mg.vcycle(b, x)
    for _ in range(2):  # the second call starts from used buffers
        xg = torch.zeros(x.shape, dtype=torch.float64, device="cuda")
        ctx.solve(torch.from_numpy(b).cuda(), xg, tol=0.0)
        got = xg.cpu().numpy()
        assert not got[:, [0, nz]].any()
        assert rel(got, x) <= 3.2e-5
    ctx.close()
