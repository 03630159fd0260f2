"""A batched update follows its context's options: changing the OC exponent
between two to_batch_step calls with the same job table gives what to_oc_update
gives with each exponent, bit for bit."""

import numpy as np
import pytest

from gpu_helpers import Ctx, dev, host, torch
from workloads import rand_density, rand_vector, small_problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind,precision", [("cantilever3d", "mixed"), ("mbb2d", "fp64")])
def test_oc_exponent_change(kind, precision):
    from paper_2205_00385_gb300 import binding as B
    p = small_problem(kind, mg_levels=2)
    rho = rand_density(p.nel, 3, 0.2, 0.8)
    t = torch()   # (the legacy stream cannot be captured)
    with t.cuda.stream(t.cuda.Stream()), Ctx(p, precision=precision) as c:
        c.set_density(rho)
        z = lambda n: dev(np.zeros(n))
        job = dict(ctx=c.ctx, rho=dev(rho), rho_phys=z(p.nel), u=dev(rand_vector(p.ndof, 4, fixed=p.fixed)),
                   dc=z(p.nel), dc_f=z(p.nel), dv_f=dev(np.ones(p.nel)), compliance_dev=z(1),
                   change_dev=z(1), volfrac=0.5, move=0.2)
        out = {}
        for eta in (0.5, 0.3, 0.5):
            B.to_oc_options(c.ctx, eta)
            job["rho"].copy_(dev(rho))
            B.to_batch_step([job], B.TO_PHASE_UPDATE, c.stream.cuda_stream)
            t.cuda.synchronize()
            got = host(job["rho"]).copy()
            rd = dev(rho)
            B.to_oc_update(c.ctx, 0.5, 0.2, job["dc_f"], job["dv_f"], rd, z(1))
            assert np.array_equal(got, host(rd)), eta
            assert np.array_equal(got, out.setdefault(eta, got))
        assert not np.array_equal(out[0.5], out[0.3])
