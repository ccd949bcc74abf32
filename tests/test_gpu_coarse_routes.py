"""Which form of the coarse operator a solve prepares and which kernel runs it."""
import numpy as np
import pytest

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
