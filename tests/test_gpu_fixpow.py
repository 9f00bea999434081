"""The constitutive law's fixed-point powers (csrc/fixpow.cuh) against 120-bit arithmetic.

rich_saturation with theta_s = 1, theta_r = 0 returns alpha / (alpha + |p|^beta).  Bound:
|p|^beta is within 2^-53 + 1.1 beta 2^-57 + 2^-58 relative, the sum, the reciprocal (1 ulp)
and the product add 4 x 2^-53 at most, so S is within (5 + 1.1 beta / 16) 2^-53 + 2^-58 of
its value; outside the domain (|p| beyond 2^+-30, beta >= 32) pow() serves, inside the wider
bound stated there."""
import dataclasses

import numpy as np
import pytest

from paper_2112_05051_gb300 import synth

torch = pytest.importorskip("torch")
mpmath = pytest.importorskip("mpmath")
pytestmark = pytest.mark.gpu


def _points():
    rng = np.random.default_rng(3)
    p = [2.0 ** rng.uniform(-29.9, 29.9, 400), rng.uniform(1.0, 80.0, 600)]
    # table cells' ends, powers of two, the ends of the domain and just outside it
    ends = 1.0 + np.arange(257) / 256.0
    p += [ends, np.nextafter(ends, 0), 2.0 ** np.arange(-32.0, 33.0), np.nextafter(2.0 ** np.arange(-32.0, 33.0), 0)]
    return np.concatenate(p)


@pytest.mark.parametrize("beta,alpha", [(3.96, 1.611e6), (4.74, 1.0), (0.5, 1.0), (1.0, 3.0), (31.5, 2.0), (40.0, 1.0)])
def test_saturation_against_exact_powers(beta, alpha):
    from paper_2112_05051_gb300 import richards as rb
    rb.load()
    ap = _points()
    soil = dataclasses.replace(synth.Soil(), alpha=alpha, beta=beta, theta_s=1.0, theta_r=0.0)
    ctx = rb.Context(synth.Grid(len(ap), 1, 1), soil, synth.infiltration_bc(), 0)
    s = torch.empty(len(ap), dtype=torch.float64, device="cuda")
    ctx.saturation(torch.tensor(-ap, device="cuda"), s)
    got = s.cpu().numpy()
    ctx.close()
    with mpmath.workprec(120):
        for x, g in zip(ap, got):
            ref = alpha / (alpha + mpmath.mpf(float(x)) ** mpmath.mpf(beta))
            tol = (5 + 1.1 * beta / 16) * 2.0 ** -53 + 2.0 ** -58
            if not (2.0 ** -30 <= x < 2.0 ** 30 and beta < 32):
                tol += (beta * abs(float(np.log(x))) + 8) * 2.0 ** -53
            if float(ref) < 1e-290:
                continue
            assert abs((mpmath.mpf(float(g)) - ref) / ref) <= tol, (x, beta)


def test_law_at_special_pressures():
    """p >= 0, -0.0 and NaN take the saturated branch; -inf and tiny heads as before."""
    from paper_2112_05051_gb300 import richards as rb
    rb.load()
    soil = synth.Soil()
    p = np.array([0.0, -0.0, 5.0, np.nan, -np.nan, -1e-300, -5e-324, -np.inf, -1e300])
    ctx = rb.Context(synth.Grid(len(p), 1, 1), soil, synth.infiltration_bc(), 0)
    s = torch.empty(len(p), dtype=torch.float64, device="cuda")
    ctx.saturation(torch.tensor(p, device="cuda"), s)
    got = s.cpu().numpy()
    ctx.close()
    np.testing.assert_allclose(got[:7], soil.theta_s, rtol=1e-15)
    np.testing.assert_allclose(got[7:], soil.theta_r, rtol=1e-15)
