"""The reduced model at its largest basis sizes (n_carm 13 to 16, the Gram-Schmidt
kernels' widest form), against the oracle.

The PARM's columns and u_last are random and the two densities far apart, so that
all the columns of the basis are independent (the oracle's QR diagonal is above
1e-7 of the columns, its singular values away from the truncation at 1e-6).
Tolerances: those of the parity tests of the reduced model."""

import numpy as np
import pytest

from gpu_helpers import Ctx, dev, host
from oracle import fe, reanalysis, sensitivity
from workloads import rand_density, rand_vector, small_problem

pytestmark = pytest.mark.gpu

CARM_TOL = {"fp64": {"u": 1e-9, "eps": 1e-8, "C": 1e-10},
            "mixed": {"u": 1e-6, "eps": 1e-6, "C": 1e-6}}


@pytest.mark.parametrize("kind,kw", [("cantilever3d", dict(nelx=8, nely=4, nelz=4)),
                                     ("mbb2d", dict(nelx=24, nely=8))])
@pytest.mark.parametrize("m", [13, 14, 16])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_widest_bases(kind, kw, m, precision):
    from paper_2205_00385_gb300 import binding as B
    p = small_problem(kind, mg_levels=2, n_parm=16, n_carm=m, **kw)
    g, KE = fe.Grid.of(p), fe.element_stiffness(p.dim, p.nu)
    rho0, rho1 = rand_density(p.nel, 21, 0.5, 1.0), rand_density(p.nel, 22, 0.5, 1.0)
    E0, E1 = (sensitivity.simp_modulus(r, p.E0, p.Emin, p.penal) for r in (rho0, rho1))
    K, Kr = (fe.stiffness(g, E, KE, p.fixed) for E in (E1, E0))
    dK = fe.apply_bcs(fe.assemble(g, E1 - E0, KE), p.fixed, diag_fixed=0.0)
    Phi = np.stack([reanalysis.normalized(rand_vector(g.ndof, 100 + i, fixed=p.fixed))
                    for i in range(16)], axis=1)
    u_last = rand_vector(g.ndof, 5, fixed=p.fixed)
    u_ref, eps_ref, Rt = reanalysis.aarmr_solve(lambda v: K @ v, lambda v: Kr @ v, lambda v: dK @ v,
                                                p.f, u_last, Phi, m)
    with Ctx(p, precision=precision) as c:
        c.set_density(rho0)
        c.set_density(rho1)
        for i in range(16):
            B.to_parm_push(c.ctx, dev(Phi[:, i]))
        B.to_carm_build(c.ctx, dev(u_last))
        kq, k, _ = B.to_carm_info(c.ctx, m)
        u = dev(np.zeros(g.ndof))
        eps = B.to_carm_solve(c.ctx, u)
        u = host(u)
    assert (kq, k) == (m, Rt.shape[1])
    tol = CARM_TOL[precision]
    assert np.linalg.norm(u - u_ref) <= tol["u"] * np.linalg.norm(u_ref)
    assert abs(eps - eps_ref) <= tol["eps"] * eps_ref
    assert abs(p.f @ u - p.f @ u_ref) <= tol["C"] * abs(p.f @ u_ref)
