"""mg_smooth on the coarsest level, which the cycles solve directly and whose
sizes may be odd: the colour passes in place, the last plane, row or column of
an odd size left as the caller passed it.

Reference: the colour passes written out in numpy from the level's stencil.
Tolerances as for the other sweeps: 1e-12 in FP64, 1e-6 a sweep in FP32 (15
units of rounding of some 60 products a node)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1904_03808_gb300 import MG_MIXED, Context, inputs as I  # noqa: E402

MU, K = I.TABLE1["mu"], I.TABLE1["K"]

# grid -> coarsest level: odd nz (4x4x5), odd nx (5x4x4), odd ny (4x7x4), all
# odd (5x5x5), and an even one
SHAPES = {(16, 16, 20): (4, 4, 5), (20, 16, 16): (5, 4, 4), (16, 28, 16): (4, 7, 4),
          (40, 40, 40): (5, 5, 5), (16, 24, 16): (4, 6, 4)}


def colour_pass(S, b, x, colour):
    nz, ny, nx = x.shape[1] - 1, x.shape[2], x.shape[3]
    pi, pj, pk = colour & 1, colour >> 1 & 1, colour >> 2
    for k in range(1 if pk else 2, nz - (nz & 1), 2):
        for j in range(pj, ny - (ny & 1), 2):
            for i in range(pi, nx - (nx & 1), 2):
                f = b[:, k, j, i].copy()
                for d in range(27):
                    if d != 13:
                        q = x[:, k + d // 9 - 1, (j + d // 3 % 3 - 1) % ny, (i + d % 3 - 1) % nx]
                        f -= S[d] @ q
                x[:, k, j, i] = np.linalg.solve(S[13], f)


@pytest.mark.parametrize("shape", list(SHAPES))
@pytest.mark.parametrize("sweeps,descending", [(1, False), (2, True), (3, False)])
@pytest.mark.parametrize("dtype,tol", [(np.float64, 1e-12), (np.float32, 1e-6)])
def test_coarsest_level(shape, sweeps, descending, dtype, tol):
    rng = np.random.default_rng(12)
    ctx = Context(*shape, 2e-2 / shape[0], K, MU, precision=MG_MIXED)
    l = ctx.levels - 1
    nx, ny, nz = ctx.level_dims(l)
    assert (nx, ny, nz) == SHAPES[shape]
    x, b = (rng.uniform(-1, 1, (3, nz + 1, ny, nx)).astype(dtype) for _ in range(2))
    xg, bg = torch.from_numpy(x.copy()).cuda(), torch.from_numpy(b).cuda()
    # whatever the level's buffers hold from before must not reach x
    ctx.smooth(l, bg, torch.full_like(xg, 1e3), 1)
    ctx.smooth(l, bg, xg, sweeps, descending)
    S, want, b64 = ctx.level_stencil(l), x.astype(np.float64), b.astype(np.float64)
    for _ in range(sweeps):
        for c in range(7, -1, -1) if descending else range(8):
            colour_pass(S, b64, want, c)
    got = xg.cpu().numpy().astype(np.float64)
    fixed = np.ones(x.shape, bool)
    fixed[:, 1:nz - (nz & 1), :ny - (ny & 1), :nx - (nx & 1)] = False
    assert np.array_equal(got[fixed], x[fixed])
    if dtype == np.float32:
        tol *= sweeps
    assert np.abs(got - want).max() <= tol * np.abs(want).max()
    ctx.close()
