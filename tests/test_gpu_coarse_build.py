"""The Galerkin coarse operator against the oracle's at the edges of the build's
tiles: column counts on both sides of each tile size, aggregates whose leaving and
staying sites are no whole number of chunks, extents of one (every hop leaves).

Tolerances: per hop an entry is an inner product of two vectors of norm <= 1 (a
column of P and D_h of another), so a sum in chunks of 48 products, with links and
columns rounded once, is off by at most about 80 units of rounding; eight hops meet
in the diagonal block: 640 * 2^-24 = 4e-5 in FP32, 640 * 2^-53 < 1e-12 in FP64."""
import numpy as np
import pytest

import oracle
import paper_1005_3043_gb300 as wmg
import synth
from tests._fields import rough_gauge

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nv", [1, 8, 9, 16, 17, 24, 25])
@pytest.mark.parametrize("L,B", [((4, 4, 4, 8), (2, 2, 2, 4)), ((6, 2, 4, 4), (3, 1, 4, 2)), ((8, 4, 4, 10), (4, 2, 2, 5))])
def test_coarse_operator(L, B, nv):
    if nv > 6 * np.prod(B):
        pytest.skip("more columns than entries")
    U = rough_gauge(L, seed=12)
    V0 = synth.gaussian_vectors(L, nv, 33)
    P, st = oracle.block_orthonormalize(V0, L, B)
    assert st == 0
    A = oracle.coarse_build(U, P, -0.1, L, B)
    for prec, tol in ((wmg.MG_FP64, 1e-12), (wmg.MG_FP32, 4e-5)):
        p = wmg.mg_default_params()
        for i in range(4):
            p.block[i] = B[i]
        p.nvec, p.setup_group, p.prec_inner = nv, 1, prec
        with wmg.WilsonMG(L, p) as mg:
            mg.set_links(U)
            mg.set_mass(-0.1)
            mg.set_null_vectors(V0)
            got = mg.coarse_op()
        assert np.abs(got - A).max() <= tol * max(1.0, np.abs(A).max()), prec
