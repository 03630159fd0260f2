"""The float64 finest-grid operator's fixed-point element arithmetic on inputs
that exercise its scaling: magnitudes from 1e-290 to 1e290, values of very
different size within one element, exact zeros, subnormal moduli differences,
and non-finite values (which must stay where float64 arithmetic puts them).

Reference: the oracle's float64 element products.  Tolerance: 1e-13 of the
largest entry, as for the other float64 products (order of summation)."""

import numpy as np
import pytest

from gpu_helpers import Ctx, dev, host
from oracle import fe, sensitivity
from workloads import rand_density, rand_vector, small_problem

pytestmark = pytest.mark.gpu


def _product(p, rho, x, op=0, prev=None):
    from paper_2205_00385_gb300 import binding as B
    with Ctx(p, precision="fp64") as c:
        if prev is not None:
            c.set_density(prev)
        c.set_density(rho)
        y = dev(np.zeros(p.ndof))
        B.to_apply(c.ctx, op, B.TO_PREC_FP64, dev(x), y)
        return host(y)


def _reference(p, rho, x):
    g = fe.Grid.of(p)
    E = sensitivity.simp_modulus(rho, p.E0, p.Emin, p.penal)
    return fe.stiffness(g, E, fe.element_stiffness(3, p.nu), p.fixed) @ x


@pytest.mark.parametrize("nel", [(2, 2, 2), (16, 8, 8), (30, 14, 18), (34, 16, 6)])
@pytest.mark.parametrize("scale", [1e-290, 1.0, 1e290])
@pytest.mark.parametrize("kind", ["random", "smooth", "decades"])
def test_scales(nel, scale, kind):
    p = small_problem("cantilever3d", nelx=nel[0], nely=nel[1], nelz=nel[2], mg_levels=2)
    rho = rand_density(p.nel, 5, 0.0, 1.0)
    x = rand_vector(p.ndof, 6, fixed=p.fixed)
    if kind == "smooth":
        x = (1.0 + 1e-6 * x) * (p.fixed == 0)
    elif kind == "decades":
        x = x * 10.0 ** np.random.default_rng(7).integers(-12, 1, p.ndof) * (x > -0.5)
    ref = _reference(p, rho, x)
    y = _product(p, rho, x * scale) / scale
    # the smooth field's products cancel: rounding is relative to |K| |x|
    assert np.max(np.abs(y - ref)) <= 1e-13 * max(np.max(np.abs(ref)),
                                                  np.max(np.abs(x)) if kind == "smooth" else 0.0)


def test_unchanged_elements_give_zero():
    """dK of a density that did not change is exactly zero, and of one element
    changed it is zero away from that element."""
    p = small_problem("cantilever3d", nelx=16, nely=8, nelz=8, mg_levels=3)
    rho = rand_density(p.nel, 8, 0.1, 1.0)
    x = rand_vector(p.ndof, 9, fixed=p.fixed)
    assert not np.any(_product(p, rho, x, op=2, prev=rho))
    other = rho.copy()
    other[5 + 16 * (3 + 8 * 4)] += 1e-9
    y = _product(p, rho, x, op=2, prev=other).reshape(9, 9, 17, 3)
    assert np.any(y[4:6, 3:5, 5:7])
    y[4:6, 3:5, 5:7] = 0.0
    assert not np.any(y)


@pytest.mark.parametrize("value", [np.nan, np.inf, -np.inf])
def test_non_finite_inputs_stay_local(value):
    """A non-finite value spoils the nodes of the elements that hold it, as in
    float64 arithmetic, and no others."""
    p = small_problem("cantilever3d", nelx=16, nely=8, nelz=8, mg_levels=3)
    rho = rand_density(p.nel, 10, 0.1, 1.0)
    x = rand_vector(p.ndof, 11, fixed=p.fixed)
    ref = _reference(p, rho, x).reshape(9, 9, 17, 3)
    x[3 * (8 + 17 * (4 + 9 * 4)) + 1] = value
    y = _product(p, rho, x).reshape(9, 9, 17, 3)
    near = np.zeros((9, 9, 17), bool)
    near[3:6, 3:6, 7:10] = True
    assert not np.any(np.isfinite(y[near]))
    assert np.max(np.abs(y[~near] - ref[~near])) <= 1e-13 * np.max(np.abs(ref))
