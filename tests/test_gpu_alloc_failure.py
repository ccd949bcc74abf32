"""Device memory that runs out in the middle of a call: every allocation of a run of
calls is refused in turn.  The call then returns MG_ERR_OOM (or does without the
buffer), a smaller call and the call itself succeed afterwards, and its solutions
solve their systems.  A size recorded before the buffer it describes, or one buffer
of a pair, would send the calls after the refusal through a null pointer."""
import numpy as np
import pytest

import oracle
import paper_1005_3043_gb300 as wmg
import synth
from tests._fields import rough_gauge

pytestmark = pytest.mark.gpu

MASS, TOL = 0.1, 1e-8
L, B = (8, 8, 8, 8), (4, 4, 4, 4)


def params(prec, **kw):
    p = wmg.mg_default_params()
    for i in range(4):
        p.block[i] = B[i]
    p.nvec, p.setup_group, p.setup_iters, p.tol, p.prec_inner = 8, 4, 1, TOL, prec
    p.delta = 0.0 if prec == wmg.MG_FP64 else 1e-4
    for k, v in kw.items():
        setattr(p, k, v)
    return p


# (precision, parameters, the steps after the setup): the basis of the GMRES smoother and the
# vectors of the MR smoother, in FP32 and FP16 storage, the coarse operator on chip, in global
# memory (coarse_kernel 1) and in the batched kernel, each with its red-black form
CASES = {
    "gmres_fp32": (wmg.MG_FP32, dict(smoother=1, smoother_steps=6, coarse_kernel=1), ("batch", "one", "more", "one")),
    "mr_fp32": (wmg.MG_FP32, dict(smoother=0), ("batch", "one", "eo32", "eo64")),
    "gmres_fp16": (wmg.MG_FP16, dict(smoother=1, smoother_steps=6, smoother_fp16=1, coarse_kernel=1),
                   ("one", "more", "batch")),
    "mr_fp16": (wmg.MG_FP16, dict(smoother=0, smoother_fp16=1, coarse_kernel=4), ("one", "batch")),
    "gmres_fp64": (wmg.MG_FP64, dict(smoother=1, smoother_steps=6), ("one", "more")),
}


@pytest.mark.parametrize("name", CASES)
def test_calls_after_a_refused_allocation(name):
    prec, kw, steps = CASES[name]
    U = rough_gauge(L, seed=8)
    V0 = synth.gaussian_vectors(L, 8, 97)
    b = np.stack([synth.gaussian_spinor(L, 98, stream=i) for i in range(6)])
    solves = lambda x, i: np.linalg.norm(b[i] - oracle.dslash(U, x, MASS, L)) <= 2 * TOL * np.linalg.norm(b[i])   # noqa: E731

    def step(mg, what, small):
        """The call, or a smaller one of its kind."""
        p = params(prec, **kw)
        if what == "more":
            p.smoother_steps = 3 if small else 9
        mg.set_params(p)
        if what == "setup":
            mg.setup(V0)
            return []
        if what == "batch":
            x = mg.solve_batched(b[:2] if small else b)[0]
        elif what.startswith("eo"):
            x = [mg.solve_eo_cg(b[0], tol=TOL, prec=wmg.MG_FP64 if what == "eo64" else wmg.MG_FP32)[0]]
        else:
            x = [mg.solve(b[0])[0]]
        return list(x)

    nth = refused = 0
    while True:
        nth += 1
        assert nth < 500
        with wmg.WilsonMG(L, params(prec, **kw)) as mg:
            mg.set_links(U)
            mg.set_mass(MASS)
            wmg.mg_fail_allocation(mg.ctx, nth)
            for what in ("setup",) + steps:
                try:
                    found = step(mg, what, False)
                except wmg.MGError as e:
                    assert e.status == wmg.MG_ERR_OOM, e
                    refused += 1
                    if what != "setup":
                        for i, x in enumerate(step(mg, what, True)):
                            assert solves(x, i), (nth, what, "small")
                    found = step(mg, what, False)
                for i in range(0, len(found), 3):
                    assert solves(found[i], i), (nth, what)
            if wmg.mg_fail_allocation(mg.ctx, 0):
                break   # fewer than nth allocations: every one has been refused once
    assert refused > 10


# (precision, coarse_kernel, lattice, aggregates, nvec): the red-black form in global memory, its
# FP16 copy, its units on chip with and without scales, and FP16 operators larger than the chip
# (76 MB, even and odd coarse extents: panels and tiles of the batched kernel)
FORMS = {"global_fp64": (wmg.MG_FP64, 0, L, B, 8), "global_fp32": (wmg.MG_FP32, 1, L, B, 8),
         "global_fp16": (wmg.MG_FP16, 1, L, B, 8), "chip_fp32": (wmg.MG_FP32, 0, L, B, 8),
         "chip_fp16": (wmg.MG_FP16, 4, L, B, 8), "panel_even": (wmg.MG_FP16, 0, (16, 16, 16, 8), (2, 2, 2, 2), 16),
         "panel_odd": (wmg.MG_FP16, 0, (12, 16, 16, 10), (2, 2, 2, 2), 16)}


@pytest.mark.parametrize("name", FORMS)
def test_solve_without_memory_for_its_fast_forms(name):
    """What a solve allocates beyond the V-cycle's buffers are faster forms of the coarse
    solve: it does without those that are refused."""
    prec, kernel, dims, block, nv = FORMS[name]
    U, b = rough_gauge(dims, seed=8), synth.gaussian_spinor(dims, 98)
    V0 = synth.gaussian_vectors(dims, nv, 97)
    p = params(prec, coarse_kernel=kernel, nvec=nv)
    for i in range(4):
        p.block[i] = block[i]
    nth, pending = 0, 0
    while not pending:
        nth += 1
        assert nth < 50
        with wmg.WilsonMG(dims, p) as mg:
            mg.set_links(U)
            mg.set_mass(MASS)
            mg.set_null_vectors(V0)
            mg.vcycle(b, prec)
            wmg.mg_fail_allocation(mg.ctx, nth)
            x, info = mg.solve(b)
            pending = wmg.mg_fail_allocation(mg.ctx, 0)
        assert info["status"] == wmg.MG_OK
        assert np.linalg.norm(b - oracle.dslash(U, x, MASS, dims)) <= 2 * TOL * np.linalg.norm(b)
    assert nth > 1
