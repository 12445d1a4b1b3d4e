"""Sweeps where the dispatch changes: FP64 strips end at 96 columns on the finest
level and at 64 on a coarse one; FP32 strips give way to the persistent rows at
128 columns in planes of nine rows and more, and on finest levels below that whose
tiles fill the chip.  Level 0 and 1 of
each grid against the oracle's colour passes: 1e-12 in FP64, 1e-6 a sweep in FP32
on the same FP32-rounded arrays (15 units of rounding of some 60 products)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle as O  # noqa: E402
from paper_1904_03808_gb300 import MG_MIXED, Context, inputs as I  # noqa: E402

MU, K = I.TABLE1["mu"], I.TABLE1["K"]
# columns of levels 0 and 1: 96/48, 98, 128/64, 132/66, and, of planes too low for
# the persistent rows, 128 and 130
SHAPES = [(96, 20, 16), (98, 8, 8), (128, 20, 16), (132, 16, 16), (256, 16, 16), (260, 16, 16)]
# finest levels below 128 columns: tiles enough for the persistent rows (80^3,
# 64x128x64, 112x64x64), too few (64^3) and a second round of few (96^3)
SHAPES += [(80, 80, 80), (64, 128, 64), (112, 64, 64), (64, 64, 64), (96, 96, 96)]


@pytest.mark.parametrize("shape", SHAPES)
def test_sweeps(shape):
    rng = np.random.default_rng(14)
    ctx = Context(*shape, 2e-2 / shape[0], K, MU, precision=MG_MIXED)
    for l in range(min(ctx.levels - 1, 2)):
        nx, ny, nz = ctx.level_dims(l)
        S = ctx.level_stencil(l)
        for dtype, tol in ((np.float64, 1e-12), (np.float32, 1e-6)):
            x, b = (rng.uniform(-1, 1, (3, nz + 1, ny, nx)).astype(dtype) for _ in range(2))
            if l:
                x[:, [0, nz]] = 0
            b64 = b.astype(np.float64)
            for sweeps, descending in ((1, False), (2, True)):
                xg, want = torch.from_numpy(x.copy()).cuda(), x.astype(np.float64)
                ctx.smooth(l, torch.from_numpy(b).cuda(), xg, sweeps, descending)
                for _ in range(sweeps):
                    for c in range(7, -1, -1) if descending else range(8):
                        O.gs_colour(S, b64, want, c)
                got = xg.cpu().numpy().astype(np.float64)
                t = tol * (sweeps if dtype == np.float32 else 1)
                assert np.array_equal(got[:, [0, nz]], x[:, [0, nz]])
                assert np.abs(got - want).max() <= t * np.abs(want).max(), (l, dtype, sweeps)
                assert np.linalg.norm(got - want) <= t * np.linalg.norm(want), (l, dtype, sweeps)
    ctx.close()


def test_large_coarse_planes_of_short_rows():
    """A coarse level of 64 x 256 nodes a plane, FP32."""
    rng = np.random.default_rng(15)
    ctx = Context(128, 512, 256, 1e-4, K, MU, precision=MG_MIXED)
    nx, ny, nz = ctx.level_dims(1)
    x, b = (rng.uniform(-1, 1, (3, nz + 1, ny, nx)).astype(np.float32) for _ in range(2))
    x[:, [0, nz]] = 0
    xg, want = torch.from_numpy(x.copy()).cuda(), x.astype(np.float64)
    ctx.smooth(1, torch.from_numpy(b).cuda(), xg, 1)
    S, b64 = ctx.level_stencil(1), b.astype(np.float64)
    for c in range(8):
        O.gs_colour(S, b64, want, c)
    got = xg.cpu().numpy().astype(np.float64)
    assert np.abs(got - want).max() <= 1e-6 * np.abs(want).max()
    ctx.close()
