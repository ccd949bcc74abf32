"""The cases by which this solver's speed is measured.

Every case is a whole call of the public interface, as a lattice program makes
it: links, random starts and sources lie on the GPU in the boundary layout, the
context is kept from call to call, and the solutions come back in device
memory.  What differs from case to case is which call (one source, a batch, a
fresh gauge field with its adaptive setup, the red-black CG), the lattice and
its aggregates, the number of near-null vectors, the inner precision and the
smoother.

Inputs: a quenched SU(3) field thermalised at beta = 6.0 by a few heatbath
sweeps on the GPU, Gaussian sources or the twelve spin-colour point sources of a
propagator.  Solves run to a true relative residual of 1e-12, so that the
solution itself is determined to about ten digits at these masses.
"""
import math

import torch

import paper_1005_3043_gb300 as wmg

BETA = 6.0
SCATTER = 0.2   # of the links that the heatbath starts from
PREC = {"fp64": wmg.MG_FP64, "fp32": wmg.MG_FP32, "fp16": wmg.MG_FP16}


def case(call, dims, nvec, prec, mass, block=(4, 4, 4, 4), **more):
    c = {"call": call, "lx": dims[0], "ly": dims[1], "lz": dims[2], "lt": dims[3], "bx": block[0], "by": block[1],
         "bz": block[2], "bt": block[3], "nvec": nvec, "prec": prec, "mass": mass, "smoother": 0, "smoother_steps": 4,
         "restart": 16, "nrhs": 1, "levels": 2, "setup_iters": 5, "point": False, "tol": 1e-12}
    c.update(more)
    return c


def listed():
    gmres = {"smoother": 1, "smoother_steps": 12}
    return [
        # the smallest configuration, plain FP64 multigrid with the default smoother, one source
        dict(case("solve", (8, 8, 8, 8), 8, "fp64", -0.75, setup_iters=3), name="solve_8_fp64"),
        # the whole job on a small field: new links, adaptive setup, one source
        dict(case("step", (8, 8, 8, 8), 8, "fp32", -0.75, setup_iters=3), name="step_8_fp32"),
        # uneven extents and aggregates, MR smoother, FP16 storage
        dict(case("solve", (12, 20, 6, 10), 10, "fp16", -0.7, block=(3, 4, 3, 5), setup_group=2), name="solve_ragged_fp16"),
        # plain FP64 multigrid on a middle lattice
        dict(case("solve", (12, 12, 12, 24), 12, "fp64", -0.7, **gmres), name="solve_12_fp64"),
        # the flagship call: one source on a light mass, FP16 storage
        dict(case("solve", (16, 16, 16, 32), 20, "fp16", -0.79, **gmres), name="solve_16_fp16"),
        # the same without FP16 storage
        dict(case("solve", (16, 16, 16, 32), 20, "fp32", -0.79, **gmres), name="solve_16_fp32"),
        # a new gauge field: links, setup at the lightest mass, a source at two masses
        dict(case("step", (16, 16, 16, 32), 20, "fp16", -0.79, mass2=-0.75, **gmres), name="step_16_fp16"),
        # a propagator: the twelve spin-colour point sources together
        dict(case("batch", (16, 16, 16, 32), 16, "fp16", -0.75, nrhs=12, point=True, **gmres), name="propagator_16_fp16"),
        # many stochastic sources on a small lattice
        dict(case("batch", (8, 8, 8, 16), 8, "fp32", -0.6, nrhs=21, smoother=1, smoother_steps=6), name="batch_8_fp32"),
        # a lattice whose coarse operator does not fit on chip
        dict(case("solve", (24, 24, 24, 32), 24, "fp16", -0.79, restart=8, **gmres), name="solve_24_fp16"),
        # the three-level W-cycle
        dict(case("solve", (16, 16, 16, 32), 20, "fp16", -0.79, levels=3, **gmres), name="solve_16_three_level"),
        # red-black CG, the solver multigrid is compared with (and used at heavy masses)
        dict(case("eo_cg", (16, 16, 16, 32), 20, "fp32", -0.7), name="eo_cg_16_fp32"),
    ]


def draw(rng):
    call = rng.choice(["solve", "solve", "step", "batch", "batch", "eo_cg"])
    prec = rng.choice(["fp16", "fp16", "fp32", "fp64"]) if call == "solve" else rng.choice(["fp16", "fp32"])
    most = {"solve": {"fp64": 1.0e4, "fp32": 1.31e5, "fp16": 1.31e5}[prec], "step": 4.0e4, "batch": 5.0e4, "eo_cg": 1.31e5}[call]
    volume = math.exp(rng.uniform(math.log(2.0e3), math.log(most)))
    if call == "eo_cg":   # even extents; the aggregates play no part
        while True:
            dims = [2 * rng.randint(2, 12) for _ in range(3)] + [2 * rng.randint(2, 20)]
            if 0.6 * volume <= math.prod(dims) <= min(1.5 * volume, most):
                return case(call, dims, 4, prec, round(rng.uniform(-0.75, -0.3), 3), block=(1, 1, 1, 1))
    while True:
        block = [rng.choice([3, 4, 4, 4]) for _ in range(4)]
        cells = [rng.randint(1, 6) for _ in range(3)] + [rng.randint(2, 9)]
        dims = [b * n for b, n in zip(block, cells)]
        if 0.6 * volume <= math.prod(dims) <= min(1.5 * volume, most) and math.prod(cells) >= 8:
            break
    nvec = rng.choice([8, 16, 24] if call == "batch" else [6, 8, 10, 12, 16, 18, 20, 24])
    more = {"setup_group": 2 if nvec % 4 else 4, "setup_iters": rng.randint(2, 4)}
    if rng.random() < 0.7:
        more.update(smoother=1, smoother_steps=rng.randint(4, 14))
    if call == "batch":
        most_rhs = min(20, 1.5e5 / volume)
        more["nrhs"] = int(math.exp(rng.uniform(math.log(2), math.log(max(3.5, most_rhs)))))
    if call == "step" and rng.random() < 0.5:
        more["mass2"] = round(rng.uniform(-0.45, -0.3), 3)
    return case(call, dims, nvec, prec, round(rng.uniform(-0.7, -0.5), 3), block=block,
                restart=rng.choice([8, 16]), **more)


# ---------------------------------------------------------------- inputs
def dims_of(c):
    return c["lx"], c["ly"], c["lz"], c["lt"]


def su2_heatbath(w, kb, gen):
    """SU(2) elements (quaternions, last axis 4) of weight exp(kb a0) about the
    direction w, by three Kennedy-Pendleton tries; the identity where all fail."""
    n = w.shape[:-1]
    a0 = torch.full(n, 2.0, device=w.device)
    for _ in range(3):
        r = torch.rand((4,) + n, generator=gen, device=w.device).clamp_min_(1e-12)
        d = -(r[0].log() + (2 * math.pi * r[1]).cos() ** 2 * r[2].log()) / kb
        a0 = torch.where((a0 > 1.5) & (r[3] ** 2 <= 1 - 0.5 * d), 1 - d, a0)
    kept = a0 > 1.5
    a0 = torch.where(kept, torch.ones_like(a0), a0)
    v = torch.randn(n + (3,), generator=gen, device=w.device)
    v = v / v.norm(dim=-1, keepdim=True) * (1 - a0 * a0).clamp_min(0).sqrt()[..., None]
    a = torch.cat([a0[..., None], v], -1)
    # a * w^dagger as quaternions
    w0, wv, av = w[..., :1], -w[..., 1:], a[..., 1:]
    g = torch.cat([a[..., :1] * w0 - (av * wv).sum(-1, keepdim=True),
                   a[..., :1] * wv + w0 * av - torch.linalg.cross(av, wv)], -1)
    one = torch.zeros_like(g)
    one[..., 0] = 1
    return torch.where(kept[..., None], one, g)


def unitary(u):
    """Gram-Schmidt on the rows and unit determinant, in 64 bits."""
    u = u.to(torch.complex128)
    a = u[..., 0, :] / u[..., 0, :].norm(dim=-1, keepdim=True)
    b = u[..., 1, :] - a * (a.conj() * u[..., 1, :]).sum(-1, keepdim=True)
    b = b / b.norm(dim=-1, keepdim=True)
    return torch.stack([a, b, torch.linalg.cross(a, b).conj()], -2)


def mul(a, b):
    """Products of many 3 x 3 matrices."""
    return (a[..., :, :, None] * b[..., None, :, :]).sum(-2)


def gauge_field(dims, gen, sweeps=7):
    """Links [mu][site][3][3], thermalised from links scattered about unity."""
    shape = tuple(reversed(dims))
    h = torch.randn((4,) + shape + (3, 3, 2), generator=gen, device="cuda")
    h = torch.view_as_complex(h)
    h = h - h.mH
    tr = torch.diagonal(h, dim1=-2, dim2=-1).sum(-1)[..., None, None] / 3
    h = SCATTER * (h - tr * torch.eye(3, device="cuda"))
    u = unitary(torch.eye(3, device="cuda") + h + mul(h, h) / 2).to(torch.complex64)
    parity = sum(torch.meshgrid(*[torch.arange(n, device="cuda") for n in shape], indexing="ij")) % 2
    axis = lambda mu: 3 - mu   # noqa: E731  site arrays run t, z, y, x
    ahead = lambda f, mu: f.roll(-1, axis(mu))   # noqa: E731
    for _ in range(sweeps):
        for mu in range(4):
            for par in range(2):
                staples = 0
                for nu in range(4):
                    if nu == mu:
                        continue
                    uv, um = u[nu], u[mu]
                    side = ahead(uv, mu)
                    up = mul(side, mul(uv, ahead(um, nu)).mH)
                    down = mul(mul(um, side).mH, uv)
                    # the lower staple starts one site back along nu
                    staples = staples + up + down.roll(1, axis(nu))
                for i, j in ((0, 1), (1, 2), (0, 2)):
                    m = mul(u[mu], staples)
                    w = torch.stack([(m[..., i, i] + m[..., j, j]).real, (m[..., i, j] + m[..., j, i]).imag,
                                     (m[..., i, j] - m[..., j, i]).real, (m[..., i, i] - m[..., j, j]).imag], -1) / 2
                    k = w.norm(dim=-1).clamp_min(1e-6)
                    q = su2_heatbath(w / k[..., None], 2 * BETA / 3 * k, gen)
                    g = torch.eye(3, device="cuda", dtype=torch.complex64).repeat(k.shape + (1, 1))
                    g[..., i, i], g[..., j, j] = torch.complex(q[..., 0], q[..., 3]), torch.complex(q[..., 0], -q[..., 3])
                    g[..., i, j], g[..., j, i] = torch.complex(q[..., 2], q[..., 1]), torch.complex(-q[..., 2], q[..., 1])
                    u[mu] = torch.where((parity == par)[..., None, None], mul(g, u[mu]), u[mu])
        u = unitary(u).to(torch.complex64)
    return unitary(u).reshape(4, -1, 3, 3).contiguous()


def gaussian(n, volume, gen):
    return torch.randn((n, volume, 4, 3), generator=gen, device="cuda", dtype=torch.complex128)


def inputs(c, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    dims = dims_of(c)
    volume = math.prod(dims)
    links = gauge_field(dims, gen)
    starts = gaussian(c["nvec"], volume, gen) if c["call"] != "eo_cg" else None
    if c["point"]:
        b = torch.zeros((c["nrhs"], volume, 4, 3), device="cuda", dtype=torch.complex128)
        site = int(torch.randint(volume, (1,), generator=gen, device="cuda"))
        for i in range(c["nrhs"]):
            b[i, site, i // 3 % 4, i % 3] = 1
    else:
        b = gaussian(c["nrhs"], volume, gen)
    return links, starts, b


def masses(c):
    return [c["mass"]] + ([c["mass2"]] if "mass2" in c else [])


# ---------------------------------------------------------------- the calls
def params(c):
    p = wmg.mg_default_params()
    for i, k in enumerate("xyzt"):
        p.block[i] = c["b" + k]
    p.nvec = c["nvec"]
    p.setup_group = c.get("setup_group", 4)
    p.setup_iters = c["setup_iters"]
    p.gcr_restart = c["restart"]
    p.tol = c["tol"]
    p.prec_inner = PREC[c["prec"]]
    p.delta = 0.0 if c["prec"] == "fp64" else 1e-4
    p.smoother = c["smoother"]
    p.smoother_steps = c["smoother_steps"]
    p.levels = c["levels"]
    return p


def prepare(c, seed):
    links, starts, b = inputs(c, seed)
    mg = wmg.WilsonMG(dims_of(c), params(c))
    x = torch.empty((len(masses(c)),) + tuple(b.shape), device="cuda", dtype=torch.complex128)
    s = {"case": c, "mg": mg, "b": b, "x": x}
    if c["call"] == "step":
        s.update(links=links, starts=starts)
        return s
    mg.set_links_device(links)
    mg.set_mass(c["mass"])
    if c["call"] != "eo_cg":
        mg.setup_device(starts)
    if c["levels"] == 3:
        gen = torch.Generator().manual_seed(seed + 1)
        mg.setup_level2(torch.randn((mg.params.nvec2, mg.Vc, mg.nc), generator=gen, dtype=torch.complex128).numpy())
    return s


def done(*infos):
    for i in infos:
        if i["status"] != wmg.MG_OK:
            raise RuntimeError("no solution: %s" % i)


def run(s):
    c, mg, b, x = s["case"], s["mg"], s["b"], s["x"]
    if c["call"] == "step":
        mg.set_links_device(s["links"])
        mg.set_mass(c["mass"])
        mg.setup_device(s["starts"])
        for i, m in enumerate(masses(c)):
            mg.set_mass(m)
            done(mg.solve_device(b[0], x[i, 0]))
    elif c["call"] == "batch":
        done(*mg.solve_batched_device(b, x, c["nrhs"]))
    elif c["call"] == "eo_cg":
        done(mg.solve_eo_cg_device(b[0], x[0, 0], tol=c["tol"], prec=PREC[c["prec"]]))
    else:
        done(mg.solve_device(b[0], x[0, 0]))
    return [v for m in x for v in m]


def work(c):
    """Bytes: links, sources, starts or the level that the call is given, each
    once, and the solutions.  Flops: one application of the operator of eq. 2
    per source, the least that a solution can be checked with."""
    volume, cells = math.prod(dims_of(c)), math.prod(c["l" + k] // c["b" + k] for k in "xyzt")
    n = c["nrhs"] * len(masses(c))
    real = 8 if c["prec"] == "fp64" else 4
    size = volume * (36 * 2 * real + n * 2 * 192)
    if c["call"] == "step":
        size += volume * (36 * 16 + c["nvec"] * 192)
    elif c["call"] != "eo_cg":
        size += volume * c["nvec"] * 24 * real
        size += cells * 9 * (2 * c["nvec"]) ** 2 * 2 * (2 if c["prec"] == "fp16" else real)
    return {"bytes": size, "flops": 1320 * volume * n}


# ---------------------------------------------------------------- 64-bit solutions in plain torch
# gamma_mu in the DeGrand-Rossi basis has an upper right 2x2 block, its adjoint below left, with one
# entry a row: (gamma psi)_i = phase[i] psi_{2 + column[i]} for i = 0, 1
GAMMA = [([1j, 1j], [1, 0]), ([-1, 1], [1, 0]), ([1j, -1j], [0, 1]), ([1, 1], [0, 1])]


def wilson(c, links, mass):
    """D of eq. 2 as a function on [site][4][3], antiperiodic in t."""
    shape = tuple(reversed(dims_of(c)))
    ahead, back, phase = [], [], []
    for mu in range(4):
        u = links[mu].reshape(shape + (3, 3)).clone()
        if mu == 3:
            u[-1] *= -1
        ahead.append(u[..., None, :, :].contiguous())
        back.append(u.roll(1, 3 - mu).mH[..., None, :, :].contiguous())
        phase.append(torch.tensor(GAMMA[mu][0], device="cuda", dtype=torch.complex128)[:, None])

    def apply(psi):
        p = psi.reshape(shape + (4, 3))
        out = (4 + mass) * p
        for mu in range(4):
            for sign, u, shift in ((-1, ahead[mu], -1), (1, back[mu], 1)):
                q = p.roll(shift, 3 - mu)
                lower = q[..., 2:, :].flip(-2) if GAMMA[mu][1][0] else q[..., 2:, :]
                h = q[..., :2, :] + sign * phase[mu] * lower
                h = 0.5 * (u[..., 0] * h[..., 0:1] + u[..., 1] * h[..., 1:2] + u[..., 2] * h[..., 2:3])
                out[..., :2, :] -= h
                h = sign * phase[mu].conj() * h
                out[..., 2:, :] -= h.flip(-2) if GAMMA[mu][1][0] else h
        return out.reshape(psi.shape)

    return apply


def solution(apply, b, tol=2e-14, most=3000):
    """BiCGStab, restarted from the true residual; None if it stalls."""
    x, r = torch.zeros_like(b), b.clone()
    size = b.norm()
    dot = lambda u, v: torch.vdot(u.reshape(-1), v.reshape(-1))   # noqa: E731
    used = 0
    for _ in range(12):
        start = r.norm()
        r0, p, rho = r.clone(), r.clone(), dot(r, r)
        while used < most:
            v = apply(p)
            alpha = rho / dot(r0, v)
            s = r - alpha * v
            t = apply(s)
            omega = dot(t, s) / dot(t, t)
            x = x + alpha * p + omega * s
            r = s - omega * t
            used += 1
            new = dot(r0, r)
            p = r + new / rho * alpha / omega * (p - omega * v)
            rho = new
            if used % 10 == 0 and float(r.norm()) < max(float(tol * size) / 2, 1e-6 * float(start)):
                break
        r = b - apply(x)
        if float(r.norm()) <= tol * float(size):
            return x
    return x if float(r.norm()) <= 2e-13 * float(size) else None


def exact(c, seed):
    """The first source's solution at each mass (the others take as long again).
    None on the large lattices at light masses, where BiCGStab stalls."""
    if math.prod(dims_of(c)) > 50000 and c["mass"] < -0.76:
        return None
    links, _, b = inputs(c, seed)
    found = [solution(wilson(c, links, m), b[0]) for m in masses(c)]
    if any(x is None for x in found):
        return None
    return [x if i == 0 else None for x in found for i in range(c["nrhs"])]
