"""The STZ rate's pair of exponentials, exp(x + y) + exp(y - x), whose second
term is formed in FP32 where it is below 1.1e-12 of the first.

The constants make beta, the prefactor and the yield factor one, and x and y are
multiples of 2^-22, so every argument is exact and D^pl is the pair itself.  A
second state with x + 288, y - 288 gives the first exponential alone (the other is
exp(-577) of it), as the kernel computes it; the pair must then lie within half a
unit of the last place (its rounding), 0.011 (an FP32 term: rounding of 2 x to
2^-20 and of expf to 2^-23, times exp(-27.6), against half a unit, 2^-53) and 0.003
(an FP64 one: a unit of exp(-6)) of the exact sum."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1904_03808_gb300 import Context, inputs as I  # noqa: E402


def rate(x, ez):
    n = x.shape[0]
    stz = dict(tau0=0.5, eps0=1.0, c0=1.0, Delta_K=0.0, Omega=1.0, T=1.0, chi_inf=1.0, ez_K=ez,
               sY=0.0, l=1.0, kB=1.0)
    bc = dict(kind=0, U_B=0.0, t_ramp=1.0, omega=0.0, R=0.3, lambda_w=1.0)
    ctx = Context(n, n, n, 1e-3, I.TABLE1["K"], I.TABLE1["mu"], bc=bc, stz=stz)
    z = lambda *s: torch.zeros(s, dtype=torch.float64, device="cuda")  # noqa: E731
    sig, out, D, sb = z(6, n, n, n), z(6, n, n, n), z(n, n, n), z(n, n, n)
    sig[4] = torch.from_numpy(x).cuda()
    ctx.stress_predict(z(3, n + 1, n, n), sig, z(n, n, n) + 1.0, 1e-3, out, D, sb)
    ctx.close()
    assert np.array_equal(sb.cpu().numpy(), x)
    return D.cpu().numpy()


@pytest.mark.parametrize("lo,hi", [(3.0, 12.5), (12.5, 13.0), (13.0, 13.8), (13.8, 14.2),
                                   (14.2, 25.0)])
def test_pair_of_exponentials(lo, hi):
    rng = np.random.default_rng(21)
    x = np.rint(rng.uniform(lo, hi, (32, 32, 32)) * 2 ** 22) / 2 ** 22
    got, first = rate(x, 32.0), rate(x + 288.0, 320.0)
    second = np.exp((-32.0 - x).astype(np.longdouble))
    err = np.abs((got.astype(np.longdouble) - first) - second) / np.spacing(got)
    assert err.max() <= 0.515
