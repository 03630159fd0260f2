"""The 3D filter (streamed layers for radii up to 3 elements, the offset list
beyond) and the mixed compliance sensitivity (streamed element columns) on
grids thinner than the filter, around the kernels' 32 x 4 tiles and
over several z-chunks, against the oracle.

Tolerances: the filter's sums of positive terms of one sign, 1e-12 relative
as in the parity test; element energies in double-float, 2^-44 of
|KE| |u_e|^2 (a few dozen roundings of 2^-48)."""

import numpy as np
import pytest

from gpu_helpers import Ctx, dev, host
from oracle import fe, filters, sensitivity
from workloads import rand_density, rand_vector, small_problem

pytestmark = pytest.mark.gpu

GRIDS = [(2, 2, 2), (4, 2, 6), (32, 8, 4), (34, 10, 6), (62, 18, 6), (4, 12, 40)]


@pytest.mark.parametrize("nel", GRIDS)
@pytest.mark.parametrize("rmin", [0.9, 1.0, 1.2, 1.5, 2.0, 2.3, 2.5, 3.0, 3.1])
def test_filter(nel, rmin):
    from paper_2205_00385_gb300 import binding as B
    p = small_problem("cantilever3d", nelx=nel[0], nely=nel[1], nelz=nel[2], mg_levels=2, rmin=rmin)
    H, Hs = filters.filter_matrix(fe.Grid.of(p), rmin)
    x = rand_density(p.nel, 3) * 10.0 ** np.random.default_rng(4).integers(-9, 3, p.nel)
    with Ctx(p, precision="mixed") as c:
        out = dev(np.zeros(p.nel))
        B.to_filter(c.ctx, B.TO_FILTER_DENSITY, dev(x), out)
        assert np.max(np.abs(host(out) * Hs / (H @ x) - 1.0)) <= 1e-12
        B.to_filter(c.ctx, B.TO_FILTER_SENS, dev(-x), out)
        assert np.max(np.abs(host(out) / -(H.T @ (x / Hs)) - 1.0)) <= 1e-12


@pytest.mark.parametrize("nel", GRIDS)
def test_sensitivity(nel):
    from paper_2205_00385_gb300 import binding as B
    p = small_problem("cantilever3d", nelx=nel[0], nely=nel[1], nelz=nel[2], mg_levels=2)
    g, KE = fe.Grid.of(p), fe.element_stiffness(3, p.nu)
    rho = rand_density(p.nel, 5, 0.0, 1.0)
    u = rand_vector(p.ndof, 6)            # not zero on the fixed DOFs
    ce = sensitivity.element_energy(g, KE, u, p.fixed)
    E = sensitivity.simp_modulus(rho, p.E0, p.Emin, p.penal)
    scale = np.max(np.abs(KE)) * 24 * np.max(np.abs(u)) ** 2 * 24
    with Ctx(p, precision="mixed") as c:
        c.set_density(rho)
        C, dc = dev(np.zeros(1)), dev(np.zeros(p.nel))
        B.to_sensitivity(c.ctx, dev(u), C, dc)
        C, dc = host(C)[0], host(dc)
    assert np.max(np.abs(dc + p.penal * (p.E0 - p.Emin) * rho ** 2 * ce)) <= 2.0 ** -44 * scale * 3
    assert abs(C - E @ ce) <= 2.0 ** -44 * scale * p.nel
