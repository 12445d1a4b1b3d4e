"""Residuals add their right-hand side after the neighbour sums have cancelled
against the centre term, so that a right-hand side much smaller than the terms of
A x keeps its digits.

With x = 1 everywhere every node forms the same sum s (zero up to rounding), and
r = fl(b - s): r - b varies by no more than one rounding of |b| + |s|, eps (|b| +
|s|), with |s| read off as the mean of b - r.  Added to the neighbour sums first, b
would be rounded at their size, 2^17 times larger here.  The restriction (weights
of sum 8, six additions) is held to 8 (1 + 3) such roundings against the FP64
restriction of b."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle as O  # noqa: E402
from paper_1904_03808_gb300 import MG_MIXED, Context, inputs as I  # noqa: E402

MU, K = I.TABLE1["mu"], I.TABLE1["K"]
SMALL = 2.0 ** -17
# strips (64, 32, 20 columns and fewer), one thread a node (odd sizes below
# 40), persistent rows with a fused restriction (256 and 128 columns)
SHAPES = [(64, 64, 64), (40, 40, 40), (256, 64, 64)]


@pytest.fixture(params=SHAPES, ids=str)
def ctx(request):
    c = Context(*request.param, 2e-2 / request.param[0], K, MU, precision=MG_MIXED)
    yield c
    c.close()


def _arrays(ctx, l, dtype):
    nx, ny, nz = ctx.level_dims(l)
    rng = np.random.default_rng(l)
    b = (SMALL * rng.uniform(-1, 1, (3, nz + 1, ny, nx))).astype(dtype)
    bg = torch.from_numpy(b).cuda()
    return b.astype(np.float64), bg, torch.ones_like(bg)


def _coarse_levels(ctx):
    return range(1, ctx.levels - 1)


def _check(r, b, eps):
    e = r.cpu().numpy().astype(np.float64)[:, 1:-1] - b[:, 1:-1]
    s = np.abs(e.mean(axis=(1, 2, 3)))
    assert (np.ptp(e, axis=(1, 2, 3)) <= eps * (SMALL + 2 * s)).all()


@pytest.mark.parametrize("dtype", [np.float64, np.float32])
def test_coarse_residual(ctx, dtype):
    f = ctx.residual if dtype == np.float64 else ctx.residual32
    for l in _coarse_levels(ctx):
        b, bg, x = _arrays(ctx, l, dtype)
        r = torch.empty_like(bg)
        f(l, bg, x, r)
        _check(r, b, np.finfo(dtype).eps)


def test_coarse_restricted_residual(ctx):
    for l in _coarse_levels(ctx):
        b, bg, x = _arrays(ctx, l, np.float32)
        nx, ny, nz = ctx.level_dims(l + 1)
        bc = torch.zeros((3, nz + 1, ny, nx), dtype=torch.float32, device="cuda")
        ctx.residual_restrict32(l, bg, x, bc)
        got = bc.cpu().numpy().astype(np.float64)
        e = (got - O.restrict(b))[:, 2:-2]
        if e.size:
            s = np.abs(e.mean(axis=(1, 2, 3))) / 8
            spread = np.ptp(e, axis=(1, 2, 3))
            assert (spread <= 32 * 2.0 ** -23 * (SMALL + 2 * s)).all(), l


@pytest.mark.parametrize("dtype", [np.float64, np.float32])
def test_finest_residual(ctx, dtype):
    b, bg, x = _arrays(ctx, 0, dtype)
    r = torch.empty_like(bg)
    (ctx.residual if dtype == np.float64 else ctx.residual32)(0, bg, x, r)
    _check(r, b, np.finfo(dtype).eps)


@pytest.mark.parametrize("value", [1.1, 0.7, 1.3, 0.9])
def test_finest_residual_of_a_constant_field(ctx, value):
    """FP32 persistent rows: every pair of neighbours gives up its share of the
    centre term before it is weighted, so a constant field has no residual in u and
    v, and in w at most the rounding of the weighted z pair, 2 lp x."""
    nx, ny, nz = ctx.level_dims(0)
    x = torch.full((3, nz + 1, ny, nx), value, dtype=torch.float32, device="cuda")
    r = torch.empty_like(x)
    ctx.residual32(0, torch.zeros_like(x), x, r)
    lp = np.float32((I.lame_lambda(K, MU) + 2 * MU) / MU)
    assert not r[:2].any()
    assert float(r[2].abs().max()) <= 0.5 * np.spacing(np.float32(2 * lp * value))


@pytest.mark.parametrize("shape", [(24, 24, 24), (32, 32, 32), (32, 32, 40), (32, 32, 48)])
def test_floor_of_the_cluster_cycle(shape):
    """Ten FP32 cycles of four and four sweeps, whole grid in one cluster, towards
    the linear profile that the moving walls leave: a sweep rounds a node's sum and
    its quotient, two units; the eight sweeps after a residual leave 16, the
    cycles before them, contracting below one half, at most as many again."""
    nx, ny, nz = shape
    ctx = Context(*shape, 2e-2 / nx, K, MU, precision=MG_MIXED, nu1=4, nu2=4, max_cycles=1,
                  inner_cycles=10)
    z = torch.linspace(-1, 1, nz + 1, dtype=torch.float64, device="cuda")[:, None, None]
    v = torch.zeros((3, nz + 1, ny, nx), dtype=torch.float64, device="cuda")
    want = v.clone()
    for a, c in enumerate((1.1, 0.7, 0.9)):
        want[a] = c * z
        v[a, 0], v[a, nz] = -c, c
    ctx.solve(torch.zeros_like(v), v, tol=0.0)
    err = torch.linalg.vector_norm(v - want) / torch.linalg.vector_norm(want)
    assert float(err) <= 32 * 2.0 ** -24
    ctx.close()
