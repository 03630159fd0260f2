"""The OC update's multiplier search over the shapes its volume function takes:
a few elements and many blocks, sensitivities over many decades, elements
without sensitivity, both damping exponents, and targets that no multiplier
meets (all elements end at their upper or their lower limits).

The reference is a float64 bisection with the same stopping bracket.  Both
roots sit within the bracket's relative 1e-13 and the volume's own rounding
(the double-float sums, ~1e-13 relative); rho moves by at most lambda's
relative error times eta, so 1e-10 absolute (as in the parity test)."""

import numpy as np
import pytest

from gpu_helpers import Ctx, dev, host
from workloads import small_problem

pytestmark = pytest.mark.gpu


def _bisect(rho, dc, dv, volfrac, move, eta):
    a = rho * np.maximum(0.0, -dc / dv) ** eta
    lo, hi = np.maximum(0.0, rho - move), np.minimum(1.0, rho + move)
    l1, l2 = 0.0, 1e9
    while l2 - l1 > 1e-13 * (l1 + l2) and l2 > 1e-80:
        mid = 0.5 * (l1 + l2)
        if np.sum(dv * np.clip(a * mid ** -eta, lo, hi)) > volfrac * rho.size:
            l1 = mid
        else:
            l2 = mid
    return np.clip(a * (0.5 * (l1 + l2)) ** -eta, lo, hi)


@pytest.mark.parametrize("nel", [(2, 2), (6, 2), (64, 16), (320, 152), (1024, 800)])
@pytest.mark.parametrize("spread", [0.5, 8.0])
@pytest.mark.parametrize("eta,volume", [(0.5, "mean"), (0.3, "mean"), (0.5, "high"), (0.5, "low")])
def test_oc_update(nel, spread, eta, volume):
    from paper_2205_00385_gb300 import binding as B
    p = small_problem("mbb2d", nelx=nel[0], nely=nel[1],
                      mg_levels=2 if nel[0] < 100 else 4 if nel[0] < 400 else 6)
    rng = np.random.default_rng(nel[0] + nel[1])
    rho = rng.uniform(0.0, 1.0, p.nel) ** 2
    dc = -np.exp(rng.normal(0.0, spread, p.nel)) * (rng.uniform(size=p.nel) > 0.2)
    dc[0] = -1.0
    dv = rng.uniform(0.8, 1.2, p.nel)
    volfrac = {"mean": float(rho.mean()), "high": 1.0, "low": 1e-3}[volume]
    ref = _bisect(rho, dc, dv, volfrac, 0.2, eta)
    with Ctx(p, precision="fp64") as c:
        B.to_oc_options(c.ctx, eta)
        rd, ch = dev(rho), dev(np.zeros(1))
        B.to_oc_update(c.ctx, volfrac, 0.2, dev(dc), dev(dv), rd, ch)
        out, change = host(rd), host(ch)[0]
    assert np.max(np.abs(out - ref)) <= 1e-10
    assert abs(change - np.max(np.abs(ref - rho))) <= 1e-10
