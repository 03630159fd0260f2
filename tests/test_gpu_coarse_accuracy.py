"""Accuracy of the coarsest grid's float32 inverse: the mixed two-level V-cycle
next to a float32 V-cycle on the host with LAPACK's float32 inverse (spotrf,
spotri) of the same coarsest matrix, both against the float64 cycle with that
matrix's float64 inverse.

The matrix is the device's own, read column by column through to_level_apply (it is
formed in float32, which costs more digits than its inversion; 3D grids, because
to_level_apply sums an entry in another order than the matrix that is inverted,
which the conditioning of 2D grids brings to the inverse's own error).  Both inverses
are backward stable in float32, so their errors have the same size: the device's
at most twice LAPACK's, rms over 12 densities.  (On the host a compensated
elimination is 0.2 to 1.5 times LAPACK's, one that rounds an entry at every
product 2.6 to 13 times from n = 336 on.)"""

import numpy as np
import pytest
import scipy.linalg as sla

from gpu_helpers import Ctx, dev, host
from oracle import fe, sensitivity, solvers
from workloads import rand_density, rand_vector, small_problem

pytestmark = pytest.mark.gpu

GRIDS = [
    ("cantilever3d", dict(nelx=12, nely=6, nelz=6), 336),
    ("cantilever3d", dict(nelx=14, nely=8, nelz=6), 480),
    ("cantilever3d", dict(nelx=16, nely=8, nelz=8), 675),
    ("cantilever3d", dict(nelx=20, nely=10, nelz=10), 1188),
]


class _Multigrid(solvers.Multigrid):
    """The oracle's hierarchy with a given inverse on its coarsest grid, in the
    precision of its matrices."""
    inv = None

    def vcycle(self, b, l=0):
        if l == self.levels - 1:
            return self.inv @ b
        return super().vcycle(b, l)

    def to_float32(self):
        f32 = lambda ms: [m.astype(np.float32) for m in ms]
        self.A, self.P, self.D, self.omega = f32(self.A), f32(self.P), f32(self.D), np.float32(self.omega)


@pytest.mark.parametrize("kind,kw,n", GRIDS)
def test_float32_inverse(kind, kw, n):
    from paper_2205_00385_gb300 import binding as B
    p = small_problem(kind, mg_levels=2, **kw)
    g, KE = fe.Grid.of(p), fe.element_stiffness(p.dim, p.nu)
    err = []
    with Ctx(p, precision="mixed") as c:
        z, e, y = dev(np.zeros(g.ndof)), dev(np.zeros(n)), dev(np.zeros((n, n)))
        for seed in range(12):
            rho = rand_density(g.nel, 300 + seed, 0.3, 1.0)
            r = rand_vector(g.ndof, 400 + seed, fixed=p.fixed)
            c.set_density(rho)
            B.to_vcycle(c.ctx, dev(r), z)
            for i in range(n):
                e.zero_()
                e[i] = 1.0
                B.to_level_apply(c.ctx, 1, e, y[i])
            A = host(y)
            assert np.max(np.abs(A - A.T)) <= 1e-6 * np.max(np.abs(A))
            A32 = np.tril(A).astype(np.float32)
            A = np.tril(A) + np.tril(A, -1).T
            E = sensitivity.simp_modulus(rho, p.E0, p.Emin, p.penal)
            mg = _Multigrid(g, fe.stiffness(g, E, KE, p.fixed), p.fixed, 2)
            assert mg.A[-1].shape[0] == n
            mg.inv = np.linalg.inv(A)
            ref = mg.vcycle(r)
            low = np.tril(sla.lapack.spotri(sla.lapack.spotrf(A32, lower=1)[0], lower=1)[0])
            mg.to_float32()
            mg.inv = low + np.tril(low, -1).T
            lapack = mg.vcycle(r.astype(np.float32))
            assert lapack.dtype == np.float32
            err.append([np.linalg.norm(v - ref) / np.linalg.norm(ref) for v in (host(z), lapack)])
    got, lap = np.sqrt(np.mean(np.square(err), axis=0))
    print(f"[float32 inverse {kind} n {n}] device {got:.2e} LAPACK {lap:.2e} ratio {got / lap:.2f}")
    assert got <= 2.0 * lap
