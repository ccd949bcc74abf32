"""The persistent batched coarse kernel at the edges of its shapes: K groups that
need padding (nc = 8, 24, 40), one column chunk and several, fewer and more jobs
than SMs, the widest panels; and right-hand sides of very different size, zero
among them, through the whole batched solve."""
import numpy as np
import pytest

import oracle
import paper_1005_3043_gb300 as wmg
import synth
from tests._fields import rough_gauge

pytestmark = pytest.mark.gpu


def params(nv, B, **kw):
    p = wmg.mg_default_params()
    for i in range(4):
        p.block[i] = B[i]
    p.nvec = nv
    p.setup_group = kw.pop("setup_group", min(4, nv))
    for k, v in kw.items():
        setattr(p, k, v)
    return p


@pytest.mark.parametrize("L,B,nv,nrhs", [((4, 4, 4, 8), (2, 2, 2, 2), 4, 1), ((8, 8, 8, 8), (2, 2, 2, 2), 4, 17),
                                         ((4, 4, 4, 8), (2, 2, 2, 2), 12, 40), ((8, 8, 8, 8), (4, 4, 4, 4), 20, 100),
                                         ((4, 4, 4, 8), (4, 4, 4, 4), 20, 256), ((4, 4, 4, 8), (2, 2, 2, 2), 24, 224),
                                         # several jobs per CTA in six and in three stages, fewer than directions
                                         ((8, 8, 8, 8), (2, 2, 2, 2), 24, 80), ((8, 8, 8, 8), (2, 2, 2, 2), 24, 192)])
def test_stencil_on_panels(L, B, nv, nrhs):
    """Against the oracle's stencil with the operator rounded to FP16: the operand is
    kept to 2^-22 and the FP32 sums over 9 * 2 Nv products add some 1e-6."""
    U = rough_gauge(L, seed=6)
    V0 = synth.gaussian_vectors(L, nv, 93)
    P, st = oracle.block_orthonormalize(V0, L, B)
    A = oracle.coarse_build(U, P, -0.2, L, B)
    A16 = A.real.astype(np.float16).astype(np.float64) + 1j * A.imag.astype(np.float16).astype(np.float64)
    Lc = oracle.coarse_dims(L, B)
    x = synth.gaussian(nrhs * oracle.volume(Lc) * 2 * nv, 94, 0).reshape(nrhs, -1, 2 * nv)
    with wmg.WilsonMG(L, params(nv, B)) as mg:
        mg.set_links(U)
        mg.set_mass(-0.2)
        mg.set_null_vectors(V0)
        for dag, apply in ((False, oracle.coarse_apply), (True, oracle.coarse_apply_dag)):
            y = mg.coarse_batched(x, dagger=dag, impl=0)
            for i in range(0, nrhs, max(1, nrhs // 7)):
                ref = apply(A16, x[i], Lc)
                assert np.abs(y[i] - ref).max() < 1e-5 * np.abs(ref).max(), (dag, i)


def test_sources_of_any_size():
    """Each source of a batch is its own problem: sources 2^60 apart in size all reach
    the tolerance, a zero source gives a zero solution."""
    L, B, nv = (8, 8, 8, 8), (4, 4, 4, 4), 8
    U = rough_gauge(L, seed=7)
    V0 = synth.gaussian_vectors(L, nv, 95)
    b0 = synth.gaussian_spinor(L, 96)
    b = np.stack([f * b0 for f in (1.0, 2.0 ** -30, 0.0, 2.0 ** 30)])
    with wmg.WilsonMG(L, params(nv, B, prec_inner=wmg.MG_FP32, delta=1e-4)) as mg:
        mg.set_links(U)
        mg.set_mass(0.1)
        mg.setup(V0)
        x, infos = mg.solve_batched(b)
    assert all(i["status"] == wmg.MG_OK for i in infos)
    for i in (0, 1, 3):
        assert np.linalg.norm(b[i] - oracle.dslash(U, x[i], 0.1, L)) <= 1e-10 * np.linalg.norm(b[i]), i
    assert not x[2].any()


def test_many_sources_of_a_wide_operator():
    """The whole batched solve where a stage of the pipeline is used more than once per job."""
    L, B, nv, nrhs = (8, 8, 8, 8), (2, 2, 2, 2), 24, 76
    U = rough_gauge(L, seed=7)
    V0 = synth.gaussian_vectors(L, nv, 95)
    b = np.stack([synth.gaussian_spinor(L, 96, stream=i) for i in range(nrhs)])
    with wmg.WilsonMG(L, params(nv, B, prec_inner=wmg.MG_FP16, delta=1e-4)) as mg:
        mg.set_links(U)
        mg.set_mass(0.1)
        mg.setup(V0)
        x, infos = mg.solve_batched(b)
    assert all(i["status"] == wmg.MG_OK for i in infos)
    for i in range(0, nrhs, 15):
        assert np.linalg.norm(b[i] - oracle.dslash(U, x[i], 0.1, L)) <= 1e-10 * np.linalg.norm(b[i]), i
