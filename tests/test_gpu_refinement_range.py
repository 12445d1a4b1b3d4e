"""The refinement loop scales each residual by a power of two near its norm: a
right-hand side so small that the squared norms are subnormal (norms below
1.5e-154) converges as the same one of ordinary size does.

The problem is linear and the factor a power of two, so the scaled run is the
ordinary one but for the digits the squared norms lose: with a norm of 2^-512 at
the start and tol 1e-4 the last squares are some 2^-1069 each, 5 bits, rounded to
nearest, and their sum of 1e4 and more good to 1%.  The residual is checked at
the ordinary scale."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1904_03808_gb300 import MG_MIXED, Context, inputs as I  # noqa: E402

MU, K = I.TABLE1["mu"], I.TABLE1["K"]


@pytest.mark.parametrize("n", [16, 32])
@pytest.mark.parametrize("inner", [1, 0])
def test_small_right_hand_side(n, inner):
    tol = 1e-4
    b = I.rhs_field(5, n, n, n)
    b[:, [0, n]] = 0
    s = 2.0 ** (-512 - np.frexp(np.linalg.norm(b))[1])  # norm 2^-513 .. 2^-512
    ctx = Context(n, n, n, 2e-2 / n, K, MU, precision=MG_MIXED, inner_cycles=inner, max_cycles=60)
    bg = torch.from_numpy(b).cuda()
    v = torch.zeros_like(bg)
    st, stats = ctx.solve(bg * s, v, tol=tol, raise_on_error=False)
    assert st == 0 and stats.rel_resid <= tol
    v /= s
    r = torch.empty_like(v)
    ctx.residual(0, bg, v, r)
    assert float(torch.linalg.vector_norm(r)) <= 1.01 * tol * np.linalg.norm(b)
    ctx.close()
