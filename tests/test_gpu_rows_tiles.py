"""Row-strip kernels on long rows (whole up to 512 nodes, then cut into tiles
with a halo) and on rows that are no multiple of 64, against the oracle: sweeps in
both orders, the residual, and the residual with its restriction, FP32 on the
same FP32-rounded arrays.

Shapes: whole rows of 272 and 512 nodes (one CTA an SM), tiles (544: three of
184, the last short of the row), a coarse level of 272 columns, ragged strips
(20 and 40 rows), and whole rows of 176 nodes.  Tolerances as for the other FP32
kernels: 2e-6 for two sweeps (30 units of rounding of some 60 products a node)
and for the residual with its restriction, 1e-6 for the residual."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle as O  # noqa: E402
from paper_1904_03808_gb300 import MG_MIXED, Context, inputs as I  # noqa: E402

MU, K = I.TABLE1["mu"], I.TABLE1["K"]
LAM = I.lame_lambda(K, MU)
SHAPES = [(272, 40, 32), (512, 64, 64), (544, 64, 64), (176, 20, 16)]


def rel(a, b):
    d = (a - b).ravel()
    return max(np.linalg.norm(d) / np.linalg.norm(b.ravel()), np.abs(d).max() / np.abs(b).max())


@pytest.mark.parametrize("shape", SHAPES)
def test_tiles_match_oracle(shape):
    rng = np.random.default_rng(8)
    ctx = Context(*shape, 2e-2 / shape[0], K, MU, precision=MG_MIXED)
    mg = O.MG(*shape, LAM, MU)
    g = lambda a: torch.from_numpy(a.astype(np.float32)).cuda()  # noqa: E731
    for l in range(min(ctx.levels - 1, 2)):
        nx, ny, nz = ctx.level_dims(l)
        x = rng.uniform(-1, 1, (3, nz + 1, ny, nx)).astype(np.float32).astype(np.float64)
        b = rng.uniform(-1, 1, x.shape).astype(np.float32).astype(np.float64)
        if l:
            x[:, [0, nz]] = 0
        S = mg.stencil(l)
        want = O.residual(S, b, x)
        r = torch.full(x.shape, float("nan"), device="cuda", dtype=torch.float32)
        ctx.residual32(l, g(b), g(x), r)
        assert rel(r.cpu().numpy().astype(np.float64), want) <= 1e-6
        bc = torch.zeros((3, nz // 2 + 1, ny // 2, nx // 2), dtype=torch.float32, device="cuda")
        ctx.residual_restrict32(l, g(b), g(x), bc)
        assert rel(bc.cpu().numpy().astype(np.float64), O.restrict(want)) <= 2e-6
        for descending in (False, True):
            xg, y = g(x), x.copy()
            ctx.smooth(l, g(b), xg, 2, descending)
            for _ in range(2):
                for col in (range(7, -1, -1) if descending else range(8)):
                    O.gs_colour(S, b, y, col)
            got = xg.cpu().numpy().astype(np.float64)
            assert np.array_equal(got[:, [0, nz]], x[:, [0, nz]])
            assert rel(got, y) <= 2e-6, (l, descending)
    ctx.close()


@pytest.mark.parametrize("shape,level", [((320, 256, 64), 1), ((144, 48, 32), 0),
                                         ((64, 64, 16), 1)])
def test_arrays_at_odd_words(shape, level):
    """Caller's arrays that start on any word are taken, with the result of
    aligned ones (up to the rounding of another kernel, 1e-6 as between the
    other pairs of kernels)."""
    rng = np.random.default_rng(9)
    ctx = Context(*shape, 2e-2 / shape[0], K, MU, precision=MG_MIXED)
    nx, ny, nz = ctx.level_dims(level)
    n = 3 * (nz + 1) * ny * nx
    b, x = (torch.from_numpy(rng.uniform(-1, 1, n).astype(np.float32)).cuda() for _ in range(2))
    b1, x1 = torch.empty(n + 1, device="cuda"), torch.empty(n + 1, device="cuda")
    b1[1:] = b
    x1[1:] = x
    sh = (3, nz + 1, ny, nx)
    ctx.smooth(level, b.view(sh), x.view(sh), 2, False)
    ctx.smooth(level, b1[1:].view(sh), x1[1:].view(sh), 2, False)
    assert rel(x1[1:].cpu().numpy(), x.cpu().numpy()) <= 1e-6
    ctx.close()
