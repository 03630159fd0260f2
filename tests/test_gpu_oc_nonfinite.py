"""The OC update on densities that are not numbers, of either sign bit: such an
element's limits are those of fmax(0, .) and fmin(1, .), which drop the NaN, and
its candidate takes the lower limit, so the new density is a number again."""

import numpy as np
import pytest

from gpu_helpers import Ctx, dev, host
from workloads import small_problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bits", [0x7FF8000000000000, 0xFFF8000000000000, 0xFFFFFFFFFFFFFFFF,
                                  0x7FFFFFFFFFFFFFFF])
def test_nan_density(bits):
    from paper_2205_00385_gb300 import binding as B
    p = small_problem("mbb2d", nelx=16, nely=8, mg_levels=2)
    rng = np.random.default_rng(1)
    rho = rng.uniform(0.2, 0.8, p.nel)
    rho.view(np.uint64)[37] = bits
    dc, dv = -rng.uniform(0.5, 2.0, p.nel), np.ones(p.nel)
    with Ctx(p, precision="fp64") as c:
        rd, ch = dev(rho), dev(np.zeros(1))
        B.to_oc_update(c.ctx, 0.5, 0.2, dev(dc), dev(dv), rd, ch)
        out, change = host(rd), host(ch)[0]
    assert out[37] == 0.0
    assert np.all(np.isfinite(out)) and np.isfinite(change)
