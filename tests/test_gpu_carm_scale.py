"""The reduced model of a small design change, against the oracle: its basis
columns C^i u fall by |C| = 1e-4 each, to 1e-26 of u and below, and their squares
beyond float32's exponents, in which the mixed path's pairs are held.  The basis
and the solution do not depend on the columns' scales.

The singular values of the unit-length columns are away from the truncation at
1e-6 (the last one kept and the first one dropped: 3.9e-6 | 7e-8 and 8e-6 |
1.3e-7).  Tolerances: those of the parity tests of the reduced model in mixed
precision."""

import numpy as np
import pytest

from gpu_helpers import Ctx, dev, host
from oracle import fe, reanalysis, sensitivity
from workloads import rand_density, rand_vector, small_problem

pytestmark = pytest.mark.gpu

CARM_TOL = {"u": 1e-6, "eps": 1e-6, "C": 1e-6}


@pytest.mark.parametrize("kind,kw,m", [("cantilever3d", dict(nelx=8, nely=4, nelz=4), 10),
                                       ("mbb2d", dict(nelx=24, nely=8), 8)])
def test_small_design_change(kind, kw, m):
    from paper_2205_00385_gb300 import binding as B
    p = small_problem(kind, mg_levels=2, n_parm=10, n_carm=m, **kw)
    g, KE = fe.Grid.of(p), fe.element_stiffness(p.dim, p.nu)
    rho0 = rand_density(p.nel, 21, 0.5, 1.0)
    rho1 = rho0 - 1e-4 * rand_density(p.nel, 22, 0.0, 1.0)
    E0, E1 = (sensitivity.simp_modulus(r, p.E0, p.Emin, p.penal) for r in (rho0, rho1))
    K, Kr = (fe.stiffness(g, E, KE, p.fixed) for E in (E1, E0))
    dK = fe.apply_bcs(fe.assemble(g, E1 - E0, KE), p.fixed, diag_fixed=0.0)
    Phi = np.stack([reanalysis.normalized(rand_vector(g.ndof, 100 + i, fixed=p.fixed))
                    for i in range(10)], axis=1)
    u_last = rand_vector(g.ndof, 5, fixed=p.fixed)
    u_ref, eps_ref, Rt = reanalysis.aarmr_solve(lambda v: K @ v, lambda v: Kr @ v, lambda v: dK @ v,
                                                p.f, u_last, Phi, m)
    with Ctx(p, precision="mixed") as c:
        c.set_density(rho0)
        c.set_density(rho1)
        for i in range(10):
            B.to_parm_push(c.ctx, dev(Phi[:, i]))
        B.to_carm_build(c.ctx, dev(u_last))
        _, k, _ = B.to_carm_info(c.ctx, m)
        u = dev(np.zeros(g.ndof))
        eps = B.to_carm_solve(c.ctx, u)
        u = host(u)
    print(f"[{kind}] k {k} {Rt.shape[1]} u {np.linalg.norm(u - u_ref) / np.linalg.norm(u_ref):.1e} "
          f"eps {abs(eps / eps_ref - 1):.1e} C {abs(p.f @ u / (p.f @ u_ref) - 1):.1e}")
    assert k == Rt.shape[1]
    tol = CARM_TOL
    assert np.linalg.norm(u - u_ref) <= tol["u"] * np.linalg.norm(u_ref)
    assert abs(eps - eps_ref) <= tol["eps"] * eps_ref
    assert abs(p.f @ u - p.f @ u_ref) <= tol["C"] * abs(p.f @ u_ref)
