"""The coarse solves of a solve run on the red-black Schur complement of D_c where
every coarse extent is even; the single-step V-cycle solves with D_c itself.  With
tight coarse tolerances both solve the same system: after one outer iteration GCR's
x is <D z, b> / |D z|^2 z with z the V-cycle of b.

Tolerances: at mass 1 the spectrum of D (and of D_c, a compression of it) lies
between about 1 and 9, so two solutions whose operators or residuals differ by eps
are within 2 * 10 * eps of each other; eps is the coarse tolerance in FP64 and
FP32 and the rounding of the FP16 operators, 2^-11, in FP16 and in a batch."""
import numpy as np
import pytest

import oracle
import paper_1005_3043_gb300 as wmg
import synth
from tests._fields import rough_gauge

pytestmark = pytest.mark.gpu

MASS = 1.0
SHAPES = [((8, 8, 8, 8), (4, 4, 4, 4), 4), ((4, 4, 8, 8), (2, 2, 2, 2), 6), ((8, 4, 4, 12), (2, 2, 2, 3), 8),
          ((4, 4, 4, 8), (2, 2, 2, 2), 24)]


def run(L, B, nv, prec, tol, batch=False, kernel=1):
    U = rough_gauge(L, seed=8)
    V0 = synth.gaussian_vectors(L, nv, 97)
    b = np.stack([synth.gaussian_spinor(L, 98, stream=i) for i in range(3)])
    p = wmg.mg_default_params()
    for i in range(4):
        p.block[i] = B[i]
    p.nvec, p.setup_group, p.prec_inner = nv, 2, prec
    p.coarse_tol, p.max_outer = tol, 1
    p.coarse_kernel = kernel                 # 1: the operator from global memory
    p.smoother_fp16 = 2
    with wmg.WilsonMG(L, p) as mg:
        mg.set_links(U)
        mg.set_mass(MASS)
        mg.set_null_vectors(V0)
        xs = mg.solve_batched(b)[0] if batch else [mg.solve(b[0])[0]]
        zs = [mg.vcycle(b[i], prec) for i in range(len(xs))]
    worst = 0.0
    for x, z, r in zip(xs, zs, b):
        q = oracle.dslash(U, z, MASS, L)
        ref = np.vdot(q, r) / np.vdot(q, q) * z
        worst = max(worst, np.linalg.norm(x - ref) / np.linalg.norm(ref))
    return worst


@pytest.mark.parametrize("L,B,nv", SHAPES)
@pytest.mark.parametrize("prec,tol,eps", [(wmg.MG_FP64, 1e-12, 1e-12), (wmg.MG_FP32, 1e-5, 1e-5),
                                          (wmg.MG_FP16, 1e-5, 2.0 ** -11)])
def test_schur_solve_is_the_full_solve(L, B, nv, prec, tol, eps):
    assert run(L, B, nv, prec, tol) < 20 * eps


# on chip: tensor-core products where the shape allows them (0), CUDA-core products (4);
# the last shape has several aggregates and both parities in every CTA, the first ones
# parts of one aggregate
@pytest.mark.parametrize("L,B,nv", SHAPES + [((8, 8, 8, 8), (2, 2, 2, 2), 10)])
@pytest.mark.parametrize("prec,tol,eps", [(wmg.MG_FP32, 1e-5, 1e-5), (wmg.MG_FP16, 1e-5, 2.0 ** -11)])
@pytest.mark.parametrize("kernel", [0, 4])
def test_schur_solve_on_chip(L, B, nv, prec, tol, eps, kernel):
    assert run(L, B, nv, prec, tol, kernel=kernel) < 20 * eps


@pytest.mark.parametrize("L,B,nv", [s for s in SHAPES if s[2] % 4 == 0])
def test_schur_solve_of_a_batch(L, B, nv):
    assert run(L, B, nv, wmg.MG_FP32, 1e-5, batch=True) < 20 * 2.0 ** -11


# CG on D_c itself in FP64: the operator in shared memory (all but the last shape, 92 MB),
# units that share aggregates, a last CTA with fewer units, odd coarse extents.  At mass 1
# an iteration amplifies the rounding of its two stencils, 9 nc 2^-53 < 1e-13 each, by less
# than the squared condition number, 100: four iterations stay within 1e-10.
@pytest.mark.parametrize("L,B,nv", SHAPES + [((6, 6, 6, 12), (2, 2, 2, 2), 12), ((6, 2, 4, 4), (2, 2, 2, 2), 1),
                                             ((6, 4, 4, 10), (2, 2, 2, 2), 25), ((8, 8, 8, 8), (2, 2, 2, 2), 25)])
def test_fp64_iterations_match_oracle(L, B, nv):
    U = rough_gauge(L, seed=8)
    V0 = synth.gaussian_vectors(L, nv, 97)
    P, st = oracle.block_orthonormalize(V0, L, B)
    assert st == 0
    A = oracle.coarse_build(U, P, MASS, L, B)
    Lc = oracle.coarse_dims(L, B)
    rc = synth.gaussian(oracle.volume(Lc) * 2 * nv, 8, 0).reshape(-1, 2 * nv)
    p = wmg.mg_default_params()
    for i in range(4):
        p.block[i] = B[i]
    p.nvec, p.setup_group = nv, 1
    with wmg.WilsonMG(L, p) as mg:
        mg.set_links(U)
        mg.set_mass(MASS)
        mg.set_null_vectors(V0)
        for k in (1, 4):
            ref, _, _ = oracle.cgnr(A, rc, Lc, 0.0, k)
            y, it, _ = mg.coarse_solve(rc, 0.0, k, wmg.MG_FP64)
            assert it == k
            assert np.abs(y - ref).max() <= 1e-10 * np.abs(ref).max(), k
