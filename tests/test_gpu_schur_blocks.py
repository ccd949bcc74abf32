"""The blocks of the red-black form of the coarse operator against numpy in 64 bits.

An odd aggregate's block is a solution of A_oo H = A_oe: Gauss-Jordan in FP64 leaves
each entry within a few nc 2^-53 cond(A_oo) of it, relative to the largest; 64 times
that is the bound.  The form is kept in 64 bits whatever the solver's precision: one
rounding on the way to 32 or 16 bits, as for D_c itself."""
import numpy as np
import pytest

import paper_1005_3043_gb300 as wmg
import synth
from tests._fields import rough_gauge

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [wmg.MG_FP64, wmg.MG_FP32, wmg.MG_FP16])
@pytest.mark.parametrize("L,B,nv", [((4, 4, 4, 8), (2, 2, 2, 2), 1), ((8, 8, 8, 8), (4, 4, 4, 4), 20),
                                    ((4, 4, 4, 4), (2, 2, 2, 2), 25), ((8, 4, 4, 12), (2, 2, 2, 3), 6)])
def test_blocks_in_64_bits(L, B, nv, prec):
    if prec == wmg.MG_FP16 and nv % 2:
        pytest.skip("FP16 storage needs an even nvec")
    p = wmg.mg_default_params()
    for i in range(4):
        p.block[i] = B[i]
    p.nvec, p.setup_group, p.prec_inner = nv, 1, prec
    with wmg.WilsonMG(L, p) as mg:
        mg.set_links(rough_gauge(L, seed=8))
        mg.set_mass(-0.3)
        mg.set_null_vectors(synth.gaussian_vectors(L, nv, 97))
        A, H = mg.coarse_op(), mg.schur_op()
    Lc = [l // b for l, b in zip(L, B)]
    X = np.arange(len(A))
    xc = [X % Lc[0], X // Lc[0] % Lc[1], X // (Lc[0] * Lc[1]) % Lc[2], X // (Lc[0] * Lc[1] * Lc[2])]
    odd = (sum(xc) & 1).astype(bool)
    assert np.array_equal(H[~odd][:, 0], A[~odd][:, 0]) and np.array_equal(H[~odd][:, 1:], -A[~odd][:, 1:])
    for x in np.flatnonzero(odd):
        bound = 64 * 2 * nv * 2.0 ** -53 * np.linalg.cond(A[x, 0])
        ref = np.concatenate([np.linalg.inv(A[x, 0])[None], np.linalg.solve(A[x, 0], A[x, 1:])])
        for d in range(9):
            assert np.abs(H[x, d] - ref[d]).max() <= bound * np.abs(ref[d]).max(), (x, d)


def test_odd_extents_are_refused():
    p = wmg.mg_default_params()
    p.nvec = 4
    with wmg.WilsonMG((12, 8, 8, 8), p) as mg:
        mg.set_links(rough_gauge((12, 8, 8, 8), seed=8))
        mg.set_null_vectors(synth.gaussian_vectors((12, 8, 8, 8), 4, 97))
        with pytest.raises(wmg.MGError) as e:
            mg.schur_op()
        assert e.value.status == wmg.MG_ERR_INVALID_ARG
