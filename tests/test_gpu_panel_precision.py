"""What the batched coarse kernel keeps of its operator, its operand and its sums."""
import numpy as np
import pytest

import paper_1005_3043_gb300 as wmg
import synth
from tests._fields import rough_gauge

pytestmark = pytest.mark.gpu


def context(L, B, nv, U, mass, V, t_antiperiodic=1, **kw):
    p = wmg.mg_default_params()
    for i in range(4):
        p.block[i] = B[i]
    p.nvec, p.setup_group = nv, 1
    for k, v in kw.items():
        setattr(p, k, v)
    mg = wmg.WilsonMG(L, p, t_antiperiodic)
    mg.set_links(U)
    mg.set_mass(mass)
    mg.set_null_vectors(V)
    return mg


# Each entry of the FP16 operator is off by at most 2^-12 of itself (entries down to 2^-28 of
# the largest), Gaussian columns add the errors up at random: the product is within 2^-11 of
# the 64-bit one in norm.  Links times `size` and 4 + m = m0 give entries of that size, from
# below the FP16 range to above it.
@pytest.mark.parametrize("size,m0", [(1.0, 3.7), (2.0 ** -16, 3.7 * 2.0 ** -16), (2.0 ** -30, 3.7 * 2.0 ** -30),
                                     (1.0, 2.0e5), (2.0 ** 18, 3.7 * 2.0 ** 18), (2.0 ** -8, 3.7)])
@pytest.mark.parametrize("dagger", [False, True])
def test_operator_of_any_size(size, m0, dagger):
    L, B, nv, nrhs = (4, 4, 4, 8), (2, 2, 2, 2), 8, 5
    U = size * rough_gauge(L, seed=8)
    with context(L, B, nv, U, m0 - 4.0, synth.gaussian_vectors(L, nv, 97)) as mg:
        x = synth.gaussian(nrhs * mg.Vc * mg.nc, 94, 0).reshape(nrhs, mg.Vc, mg.nc)
        y, ref = (mg.coarse_batched(x, dagger=dagger, impl=i) for i in (0, 1))
    for i in range(nrhs):
        assert np.linalg.norm(y[i] - ref[i]) <= 2.0 ** -11 * np.linalg.norm(ref[i]), i
