"""Storage of a float64 hierarchy's first coarse level: its stencil and element
matrices together take at most 8 GB, beyond which the level is applied from the
finest moduli; and that form, which only such grids use, checked on one."""

import numpy as np
import pytest

from workloads import small_problem

# grid, levels, level 1 stored
GRIDS = [((320, 160, 160), 6, True), ((352, 192, 192), 6, True), ((416, 192, 192), 6, False),
         ((512, 192, 192), 6, False), ((512, 256, 256), 7, False)]


def test_stored_level_is_at_most_8_gb():
    """Workspace of a float64 context against its mixed counterpart's arrays: 603
    bytes an element without the stored level (at one PARM and CARM column)."""
    from paper_2205_00385_gb300 import binding as B
    for nel, levels, stored in GRIDS:
        d = B.make_desc(3, nel, 1.0, 1e-9, 0.3, 3.0, 2.0, levels, B.TO_FP64, 1, 1)
        n = int(np.prod(nel))
        level1 = B.to_workspace_bytes(d) - 603 * n
        assert level1 <= 8.0e9 and (level1 > 500 * n) == stored, (nel, level1)


@pytest.mark.gpu
def test_implicit_level_beyond_the_limit():
    """416 x 192 x 192 in float64.  The Galerkin operator by its definition: for nodal
    fields a, b that are trilinear over the whole grid, and so the interpolants of
    their coarse values, a_c . A_1 b_c = a . K b.  The fields vanish at the support
    (the face x = 0).  Sums of 15 million terms in double precision, of one sign in
    the energies: 1e-11 of sqrt(E_a E_b).  Then the V-cycle M, which smooths and
    corrects symmetrically: a . M b = b . M a, to 1e-10 (the coarsest solve amplifies a
    cycle's rounding about 1e4 times here: the float32 cycle is 5e-4 off)."""
    import torch
    from gpu_helpers import Ctx, dev
    from paper_2205_00385_gb300 import binding as B
    p = small_problem("cantilever3d", nelx=416, nely=192, nelz=192, mg_levels=6, n_parm=1, n_carm=1)
    fixed = dev(p.fixed).bool()
    t = lambda n: torch.zeros(n, dtype=torch.float64, device="cuda")

    def fields(step):
        x, y, z = (torch.arange(0, m + 1, step, dtype=torch.float64, device="cuda") / m
                   for m in (p.nelx, p.nely, p.nelz))
        Z, Y, X = torch.meshgrid(z, y, x, indexing="ij")
        for f in (X, X * Y, X * Z, X * Y * Z):
            for c in range(3):
                v = torch.zeros(*X.shape, 3, dtype=torch.float64, device="cuda")
                v[..., c] = f
                yield v.reshape(-1)

    fine, coarse = list(fields(1)), list(fields(2))
    assert not any(bool((v[fixed] != 0).any()) for v in fine[:3])
    torch.manual_seed(3)
    rho = 0.2 + 0.8 * torch.rand(p.nel, dtype=torch.float64, device="cuda")
    r = torch.randn(2, p.ndof, dtype=torch.float64, device="cuda")
    with Ctx(p, precision="fp64") as c:
        B.to_set_density(c.ctx, rho)
        Kb, Ab = [], []
        for v, w in zip(fine, coarse):
            y, yc = t(p.ndof), t(w.numel())
            B.to_apply(c.ctx, B.TO_OP_K, B.TO_PREC_FP64, v, y)
            B.to_level_apply(c.ctx, 1, w, yc)
            Kb.append(y)
            Ab.append(yc)
        E = torch.stack([torch.stack([a @ y for y in Kb]) for a in fine])
        Ec = torch.stack([torch.stack([a @ y for y in Ab]) for a in coarse])
        s = E.diagonal().sqrt()
        assert float(((E - Ec).abs() / (s[:, None] * s[None, :])).max()) <= 1e-11
        del Kb, Ab, fine, coarse
        a, b = r[0] * ~fixed, r[1] * ~fixed
        Ma, Mb = t(p.ndof), t(p.ndof)
        B.to_vcycle(c.ctx, a, Ma)
        B.to_vcycle(c.ctx, b, Mb)
        aMa, bMb = a @ Ma, b @ Mb
        assert float(aMa) > 0 and float(bMb) > 0
        assert float((a @ Mb - b @ Ma).abs()) <= 1e-10 * float((aMa * bMb).sqrt())
