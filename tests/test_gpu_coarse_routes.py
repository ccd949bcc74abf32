"""Which form of the coarse operator a solve prepares and which kernel runs it."""
import numpy as np
import pytest

import oracle
import paper_1005_3043_gb300 as wmg
import synth
from tests._fields import rough_gauge

pytestmark = pytest.mark.gpu

MASS = 1.0
SMALL = ((8, 8, 8, 8), (4, 4, 4, 4), 8)
# FP16 operators that fit no chip: 76 MB with even coarse extents, 71 MB with odd ones
BIG, BIG_ODD = ((16, 16, 16, 8), (2, 2, 2, 2), 16), ((12, 16, 16, 10), (2, 2, 2, 2), 16)


def context(shape, prec, kernel, **kw):
    (L, B, nv) = shape
    p = wmg.mg_default_params()
    for i in range(4):
        p.block[i] = B[i]
    p.nvec, p.setup_group, p.prec_inner, p.coarse_kernel, p.smoother_fp16 = nv, 2, prec, kernel, 2
    for k, v in kw.items():
        setattr(p, k, v)
    mg = wmg.WilsonMG(L, p)
    mg.set_links(rough_gauge(L, seed=8))
    mg.set_mass(MASS)
    mg.set_null_vectors(synth.gaussian_vectors(L, nv, 97))
    return mg


@pytest.mark.parametrize("shape,prec,kernel,launches", [
    # the red-black blocks, their FP32 copy and the copy that the kernel reads
    (SMALL, wmg.MG_FP32, 0, 3), (SMALL, wmg.MG_FP16, 4, 3), (SMALL, wmg.MG_FP16, 1, 3), (BIG, wmg.MG_FP16, 0, 3),
    (SMALL, wmg.MG_FP64, 0, 2),
    # D_c: its copy (the tiles of the batched kernel)
    (BIG_ODD, wmg.MG_FP16, 0, 1)])
def test_a_solve_prepares_the_form_that_it_runs(shape, prec, kernel, launches):
    """After a change of the mass the first solve launches what prepares its form of the
    operator, once, and nothing for a form that it does not run."""
    b = synth.gaussian_spinor(shape[0], 98)
    with context(shape, prec, kernel, max_outer=1) as mg:
        mg.solve(b)
        counts = []
        for mass in (MASS + 0.1, None):
            if mass:
                mg.set_mass(mass)
            before = wmg.mg_kernel_launches()
            mg.solve(b)
            counts.append(wmg.mg_kernel_launches() - before)
    assert counts[0] - counts[1] == launches, counts


# 8^4 with 2^4 aggregates, Nv = 24 in FP32: 42 MB, six 32-word chunks of a thread's share, four in
# tensor memory and two in shared memory
CHUNKS = ((8, 8, 8, 8), (2, 2, 2, 2), 24)
REGISTER, TMEM, TMEM_MMA, PANEL = 0, 3, 4, 5


@pytest.mark.parametrize("shape,prec,kernel,ran,red_black", [
    (SMALL, wmg.MG_FP64, 0, REGISTER, 1), (SMALL, wmg.MG_FP32, 1, REGISTER, 1), (SMALL, wmg.MG_FP16, 1, REGISTER, 1),
    (SMALL, wmg.MG_FP32, 0, TMEM, 1), (SMALL, wmg.MG_FP16, 4, TMEM, 1),
    (SMALL, wmg.MG_FP16, 0, TMEM_MMA, 0),              # its iterations are too short for the halves' barriers
    (((12, 8, 8, 8), (4, 4, 4, 4), 8), wmg.MG_FP32, 0, TMEM, 0), (((12, 8, 8, 8), (4, 4, 4, 4), 8), wmg.MG_FP64, 0, REGISTER, 0),
    (CHUNKS, wmg.MG_FP32, 0, TMEM, 1), (BIG, wmg.MG_FP16, 0, PANEL, 1), (BIG_ODD, wmg.MG_FP16, 0, PANEL, 0),
    (BIG, wmg.MG_FP16, 1, REGISTER, 1)])
def test_kernel_and_form_of_a_solve(shape, prec, kernel, ran, red_black):
    """The kernel and form that each route takes, and that its correction is that of D_c:
    after one outer iteration x is <D z, b> / |D z|^2 z, z the V-cycle of b, which runs on
    D_c (tolerances: test_gpu_red_black_coarse.py)."""
    L = shape[0]
    tol, eps = {wmg.MG_FP64: (1e-12, 1e-12), wmg.MG_FP32: (1e-5, 1e-5), wmg.MG_FP16: (1e-5, 2.0 ** -11)}[prec]
    b = synth.gaussian_spinor(L, 98)
    with context(shape, prec, kernel, coarse_tol=tol, max_outer=1) as mg:
        assert (mg.coarse_kernel(), mg.coarse_red_black()) == (-1, -1)
        x = mg.solve(b)[0]
        assert (mg.coarse_kernel(), mg.coarse_red_black()) == (ran, red_black)
        z = mg.vcycle(b, prec)
        assert mg.coarse_red_black() == 0
    q = oracle.dslash(rough_gauge(L, seed=8), z, MASS, L)
    ref = np.vdot(q, b) / np.vdot(q, q) * z
    assert np.linalg.norm(x - ref) < 20 * eps * np.linalg.norm(ref)


@pytest.mark.parametrize("shape,red_black", [(SMALL, 1), (((12, 8, 8, 8), (4, 4, 4, 4), 8), 0)])
def test_kernel_and_form_of_a_batch(shape, red_black):
    with context(shape, wmg.MG_FP32, 0) as mg:
        b = np.stack([synth.gaussian_spinor(shape[0], 98, stream=i) for i in range(2)])
        mg.solve_batched(b)
        assert (mg.coarse_kernel(), mg.coarse_red_black()) == (PANEL, red_black)


# rows that a CTA takes in two passes: 512 aggregates in four parts, 1280 in three
@pytest.mark.parametrize("L,nv", [((8, 8, 8, 16), 16), ((8, 8, 10, 32), 6)])
def test_fp64_iterations_in_several_passes(L, nv):
    """Four CG iterations on D_c in FP64 against the oracle's (the bound and its derivation:
    test_gpu_red_black_coarse.py)."""
    B = (2, 2, 2, 2)
    U, V0 = rough_gauge(L, seed=8), synth.gaussian_vectors(L, nv, 97)
    P, st = oracle.block_orthonormalize(V0, L, B)
    assert st == 0
    A, Lc = oracle.coarse_build(U, P, MASS, L, B), oracle.coarse_dims(L, B)
    rc = synth.gaussian(oracle.volume(Lc) * 2 * nv, 8, 0).reshape(-1, 2 * nv)
    ref, _, _ = oracle.cgnr(A, rc, Lc, 0.0, 4)
    with context((L, B, nv), wmg.MG_FP64, 0) as mg:
        y, it, _ = mg.coarse_solve(rc, 0.0, 4, wmg.MG_FP64)
    assert it == 4
    assert np.abs(y - ref).max() <= 1e-10 * np.abs(ref).max()


@pytest.mark.parametrize("prec,kernel", [(wmg.MG_FP64, 0), (wmg.MG_FP32, 1), (wmg.MG_FP16, 1)])
def test_red_black_form_of_the_widest_level(prec, kernel):
    """Level 2 at Nv2 = 32, the widest operator there is (64 dof): the solve runs its
    red-black form and reaches its tolerance."""
    L = (8, 8, 8, 16)
    b = synth.gaussian_spinor(L, 98)
    kw = dict(levels=3, nvec2=32, smoother_steps1=2, tol=1e-8, delta=0.0 if prec == wmg.MG_FP64 else 1e-4)
    p = wmg.mg_default_params()
    for i in range(4):
        p.block[i] = p.block2[i] = 2
    p.nvec, p.setup_group, p.prec_inner, p.coarse_kernel = 16, 2, prec, kernel
    for k, v in kw.items():
        setattr(p, k, v)
    U = rough_gauge(L, seed=8)
    with wmg.WilsonMG(L, p) as mg:
        mg.set_links(U)
        mg.set_mass(MASS)
        mg.set_null_vectors(synth.gaussian_vectors(L, 16, 97))
        n1 = mg.Vc * mg.nc
        mg.set_level2_vectors(synth.gaussian(32 * n1, 5, 0).reshape(32, mg.Vc, mg.nc))
        x, info = mg.solve(b)
        assert (mg.coarse_kernel(), mg.coarse_red_black()) == (REGISTER, 1)
    assert info["status"] == wmg.MG_OK
    assert np.linalg.norm(b - oracle.dslash(U, x, MASS, L)) <= 2e-8 * np.linalg.norm(b)
