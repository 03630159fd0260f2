"""The OC multiplier search where the volume is nearly flat in lambda (most
elements at a limit, two clusters with the target on the plateau between them):
the secant points miss there and the search takes more sweeps than are launched
up front.

Reference: a float64 bisection, as in the search's other test (1e-10).  Where the
target lies on a plateau every multiplier of it gives the same design.  The last
test compares times: such an update takes no more than 5 times an ordinary one
(it is some 15 more sweeps of the same cost, next to filter-free passes)."""

import numpy as np
import pytest

from gpu_helpers import Ctx, dev, host, torch
from test_gpu_oc_search import _bisect
from workloads import small_problem

pytestmark = pytest.mark.gpu


def _designs(n):
    """name -> rho, dc, volume fraction (dv = 1, move 0.2)"""
    rng = np.random.default_rng(5)
    c = rng.uniform(size=n) < 0.5
    jitter = rng.uniform(0.99, 1.01, n)
    plateau = float(np.mean(np.where(c, 0.7, 0.3)))
    half, k = n // 2, np.arange(n)
    few = np.exp(rng.normal(0, 2, n))
    return {
        "plateau": (np.full(n, 0.5), -np.where(c, 1e3, 1e-3), plateau),
        "near plateau": (np.full(n, 0.5), -np.where(c, 1e3, 1e-3) * jitter, plateau - 1e-6),
        "20 active": (np.where(k < half, 0.0, np.where(k < n - 20, 1.0, 0.5)),
                      -np.where(k < half, 1e-9, np.where(k < n - 20, 1e6, few)), (half - 20 + 8.0) / n),
        "ordinary": (rng.uniform(0, 1, n) ** 2, -np.exp(rng.normal(0, 1, n)), 0.33),
    }


@pytest.mark.parametrize("nel,levels", [((8, 4, 4), 2), ((32, 16, 16), 3), ((96, 48, 48), 4)])
@pytest.mark.parametrize("eta", [0.5, 0.3])
def test_flat_volume(nel, levels, eta):
    from paper_2205_00385_gb300 import binding as B
    p = small_problem("cantilever3d", nelx=nel[0], nely=nel[1], nelz=nel[2], mg_levels=levels)
    dv = np.ones(p.nel)
    with Ctx(p, precision="mixed") as c:
        B.to_oc_options(c.ctx, eta)
        for name, (rho, dc, volfrac) in _designs(p.nel).items():
            ref = _bisect(rho, dc, dv, volfrac, 0.2, eta)
            rd, ch = dev(rho), dev(np.zeros(1))
            B.to_oc_update(c.ctx, volfrac, 0.2, dev(dc), dev(dv), rd, ch)
            # (20 active: their share of the volume resolves lambda to 1e-16 n / 20)
            tol = 1e-10 + (1e-15 * p.nel if name == "20 active" else 0.0)
            assert np.max(np.abs(host(rd) - ref)) <= tol, name
            assert abs(host(ch)[0] - np.max(np.abs(ref - rho))) <= tol


@pytest.mark.parametrize("eta", [0.5, 0.3])
def test_time_of_a_flat_volume(eta):
    from paper_2205_00385_gb300 import binding as B
    t = torch()
    p = small_problem("cantilever3d", nelx=192, nely=96, nelz=96, mg_levels=5, n_parm=1, n_carm=1)
    us = {}
    with Ctx(p, precision="mixed") as c:
        B.to_oc_options(c.ctx, eta)
        dvd, ch = dev(np.ones(p.nel)), dev(np.zeros(1))
        for name, (rho, dc, volfrac) in _designs(p.nel).items():
            r0, dcd, ts = dev(rho), dev(dc), []
            for _ in range(7):
                r, e = r0.clone(), [t.cuda.Event(enable_timing=True) for _ in range(2)]
                t.cuda.synchronize()
                e[0].record()
                B.to_oc_update(c.ctx, volfrac, 0.2, dcd, dvd, r, ch)
                e[1].record()
                t.cuda.synchronize()
                ts.append(1e3 * e[0].elapsed_time(e[1]))
            us[name] = float(np.median(ts))
    print(f"[oc flat volume, eta {eta}] us {us}")
    assert max(us.values()) <= 5.0 * us["ordinary"]
