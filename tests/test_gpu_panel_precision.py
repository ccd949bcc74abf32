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


def exact_context(L, mass, **kw):
    """D_c with entries that FP16 holds exactly: unit links, prototypes constant on each
    spin-colour component (P = 1/4 on 2^4 aggregates), a dyadic mass.  On an extent that is
    even a column of D_c then has entries on the site itself and its neighbours only."""
    V = np.zeros((4, int(np.prod(L)), 4, 3), complex)
    for i in range(4):
        V[i, :, i // 3, i % 3] = V[i, :, 2 + i // 3, i % 3] = 1.0
    return context(L, (2, 2, 2, 2), 4, synth.unit_gauge(L), mass, V, **kw)


@pytest.mark.parametrize("nrhs,bits", [(1, 23), (3, 21)])
def test_operand_keeps_its_bits(nrhs, bits):
    """Columns of one entry per neighbourhood, so that an entry of y is one product (twice
    the same entry where two neighbours are one site): y / A is the operand as the kernel
    holds it.  FP32 for a single right-hand side, 22 bits in a batch, rounded to nearest and
    the product once more, for entries down to 2^-12 of the largest."""
    with exact_context((8, 8, 8, 16), -0.5) as mg:
        A = mg.coarse_op()
        assert np.array_equal(A, A.real.astype(np.float16) + 1j * A.imag.astype(np.float16).astype(float))
        rng = np.random.default_rng(3)
        X = np.arange(mg.Vc)
        t = X // 64
        x = np.zeros((nrhs, mg.Vc, mg.nc), complex)
        x[:, 0, 0] = 1.0
        far = np.flatnonzero((X % 64 == 42) & (t == 4))[0]   # (2, 2, 2, 4), four and more hops from 0
        for k in range(13):
            for i in range(nrhs):
                v = rng.uniform(1, 2, 2).astype(np.float32).astype(float)
                x[i, far, 5] = 2.0 ** -k * (v[0] + 1j * v[1]) / 2
            y, ref = (mg.coarse_batched(x, impl=q) for q in (0, 1))
            for i in range(nrhs):
                z = np.abs(ref[i, far]) > 0
                assert z.any()
                for part in (np.real, np.imag):
                    p, q = part(y[i, far][z]), part(ref[i, far][z])
                    assert np.all(np.abs(p - q) <= 2.0 ** -bits * np.abs(q)), (k, i)


@pytest.mark.parametrize("prec,nrhs", [(wmg.MG_FP32, 1), (wmg.MG_FP32, 5), (wmg.MG_FP16, 3)])
def test_sums_of_a_low_mode(prec, nrhs):
    """The constant mode of the free periodic operator: D_c v = m v exactly, so the CG on
    D_c^dag D_c solves it in one iteration with alpha = |s|^2 / |u|^2 = m^-2 to a few times
    2^-24.  |u|^2 is 2^-40 of |r|^2; alpha off by more than the tolerance, 10^-3, takes a
    second iteration.  81 aggregates (no red-black form)."""
    L = (12, 12, 12, 12)
    rng = np.random.default_rng(5)
    V = np.zeros((4, 12 ** 4, 4, 3), complex)
    for i in range(4):
        V[i, :, i // 3, i % 3] = V[i, :, 2 + i // 3, i % 3] = 1.0
    c = rng.standard_normal((nrhs, 4, 2)) @ np.array([1, 1j])
    b = np.einsum("ni,ivsc->nvsc", c, V)
    with context(L, (4, 4, 4, 4), 4, synth.unit_gauge(L), 2.0 ** -10, V, t_antiperiodic=0, prec_inner=prec,
                 coarse_tol=1e-3, max_outer=1) as mg:
        A = mg.coarse_op()
        assert np.array_equal(A, A.real.astype(np.float16) + 1j * A.imag.astype(np.float16).astype(float))
        infos = mg.solve_batched(b)[1]
    assert [i["coarse_iters"] for i in infos] == [1] * nrhs


@pytest.mark.parametrize("mass", [-0.3, 0.2])
def test_one_source_is_as_near_to_64_bits_as_before(mass):
    """A single FP16 source whose operator exceeds the chip: the correction of the panel
    kernel (coarse_kernel 0) is as near to the FP64 one as the register-streaming kernel's
    (coarse_kernel 1).  Both round the same entries to 11 bits under a scale of the largest
    one (per aggregate, per block), so their errors are of one size; odd coarse extents: both
    run on D_c."""
    L, nv = (12, 16, 16, 10), 16
    U, b, V = rough_gauge(L, seed=8), synth.gaussian_spinor(L, 98), synth.gaussian_vectors(L, nv, 97)
    xs = []
    for prec, kernel, tol in ((wmg.MG_FP64, 0, 1e-12), (wmg.MG_FP16, 1, 1e-5), (wmg.MG_FP16, 0, 1e-5)):
        with context(L, (2, 2, 2, 2), nv, U, mass, V, prec_inner=prec, coarse_kernel=kernel, coarse_tol=tol, max_outer=1,
                     smoother_fp16=2, max_coarse=20000) as mg:
            xs.append(mg.solve(b)[0])
    register, panel = (np.linalg.norm(x - xs[0]) for x in xs[1:])
    assert panel <= 1.2 * register


@pytest.mark.parametrize("L,B", [((8, 8, 8, 16), (2, 2, 2, 2)), ((6, 8, 8, 16), (2, 2, 2, 2))])
def test_a_batch_does_not_depend_on_earlier_ones(L, B):
    """The same two sources before and after a batch of 40, bit for bit: the panels of a
    call are as wide as its own sources need."""
    U, b = rough_gauge(L, seed=8), np.stack([synth.gaussian_spinor(L, 98, stream=i) for i in range(40)])
    with context(L, B, 8, U, 0.1, synth.gaussian_vectors(L, 8, 97), prec_inner=wmg.MG_FP32, tol=1e-8) as mg:
        first = mg.solve_batched(b[:2])
        mg.solve_batched(b)
        again = mg.solve_batched(b[:2])
    assert np.array_equal(first[0], again[0])
    for i, k in zip(first[1], again[1]):
        assert i["coarse_iters"] == k["coarse_iters"]
