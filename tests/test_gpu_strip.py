"""FP64 sweeps and residuals on row strips (two launches a sweep) against the
oracle's colour passes and residual, every level with a coarser one.

Shapes: strips of 8 and of 4 rows, ragged last strips (ny = 36, 20, 12), planes
shorter than a strip's window (ny = 4, 6), the widest rows of either operator
(128 on the finest level, 64 on a coarse one) and wider ones, which take the
colour launches.  Tolerance 1e-12: FP64 rounding of some 60 products a node
over three sweeps, as for the colour launches."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle as O  # noqa: E402
from paper_1904_03808_gb300 import Context, inputs as I  # noqa: E402

MU, K = I.TABLE1["mu"], I.TABLE1["K"]
LAM = I.lame_lambda(K, MU)
SHAPES = [(64, 64, 64), (128, 36, 16), (128, 64, 48), (160, 16, 16), (20, 12, 8), (16, 4, 8),
          (16, 6, 2)]


def rel(a, b):
    d = (a - b).ravel()
    return max(np.linalg.norm(d) / np.linalg.norm(b.ravel()), np.abs(d).max() / np.abs(b).max())


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("sweeps,descending", [(1, False), (3, True)])
def test_strips_match_oracle(shape, sweeps, descending):
    rng = np.random.default_rng(4)
    ctx = Context(*shape, 2e-2 / shape[0], K, MU)
    mg = O.MG(*shape, LAM, MU)
    for l in range(max(ctx.levels - 1, 1)):
        nx, ny, nz = ctx.level_dims(l)
        x = rng.uniform(-1, 1, (3, nz + 1, ny, nx))
        b = rng.uniform(-1, 1, x.shape)
        if l:
            x[:, [0, nz]] = 0
        S = mg.stencil(l)
        xg, bg = torch.from_numpy(x.copy()).cuda(), torch.from_numpy(b).cuda()
        r = torch.full_like(xg, float("nan"))
        ctx.residual(l, bg, xg, r)
        assert rel(r.cpu().numpy(), O.residual(S, b, x)) <= 1e-12
        ctx.smooth(l, bg, xg, sweeps, descending)
        walls = x[:, [0, nz]].copy()
        for _ in range(sweeps):
            for col in (range(7, -1, -1) if descending else range(8)):
                O.gs_colour(S, b, x, col)
        got = xg.cpu().numpy()
        assert np.array_equal(got[:, [0, nz]], walls)
        assert rel(got, x) <= 1e-12, l
    ctx.close()
