"""The blocks of the red-black form of the coarse operator against numpy in 64 bits.

An odd aggregate's block is a solution of A_oo H = A_oe: Gauss-Jordan in FP64 leaves
each entry within a few nc 2^-53 cond(A_oo) of it, relative to the largest; 64 times
that is the bound.  The form is kept in 64 bits whatever the solver's precision: one
rounding on the way to 32 or 16 bits, as for D_c itself."""
import numpy as np
import pytest

import oracle
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


# Near an eigenvalue of a diagonal block the form loses its bits: the solves use D_c then.
# Solve and V-cycle run the same kernel on the same operator (see test_gpu_red_black_coarse.py
# for x), so they differ by the rounding of GCR's scalars and vector updates only.
@pytest.mark.parametrize("prec,kernel,eps", [(wmg.MG_FP64, 1, 1e-11), (wmg.MG_FP32, 1, 1e-5), (wmg.MG_FP32, 0, 1e-5),
                                             (wmg.MG_FP16, 1, 1e-5), (wmg.MG_FP16, 4, 1e-5)])
def test_nearly_singular_block_falls_back(prec, kernel, eps):
    L, nv = (4, 4, 4, 8), 8
    U, b = rough_gauge(L, seed=8), synth.gaussian_spinor(L, 98)
    p = wmg.mg_default_params()
    for i in range(4):
        p.block[i] = 2
    p.nvec, p.setup_group, p.prec_inner, p.coarse_kernel = nv, 2, prec, kernel
    p.coarse_tol, p.max_outer, p.smoother_fp16 = 1e-2, 1, 2
    with wmg.WilsonMG(L, p) as mg:
        mg.set_links(U)
        mg.set_mass(0.0)
        mg.set_null_vectors(synth.gaussian_vectors(L, nv, 97))
        A = mg.coarse_op()
        X = np.arange(len(A))
        odd = (X % 2 + X // 2 % 2 + X // 4 % 2 + X // 8) % 2 == 1
        ev = np.linalg.eigvals(A[odd, 0])
        near = ev[np.abs(ev.imag) < 1e-6].real.min()   # real up to the rounding of the FP32 products
        for gap, works in ((1.0, True), (1e-6, False)):
            mass = gap - near
            mg.set_mass(mass)
            if works:
                mg.schur_op()
                continue
            with pytest.raises(wmg.MGError) as e:
                mg.schur_op()
            assert e.value.status == wmg.MG_ERR_NUMERIC
            x, z = mg.solve(b)[0], mg.vcycle(b, prec)
            q = oracle.dslash(U, z, mass, L)
            ref = np.vdot(q, b) / np.vdot(q, q) * z
            assert np.linalg.norm(x - ref) <= eps * np.linalg.norm(ref)
