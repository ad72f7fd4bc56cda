"""Timed cases of the overlap-fermion library: what a lattice-QCD program has it do.

Each case goes through the package's public Python entry points (`Context`, `Field`).  The kinds:

  hw       load a canonical source into an internal field, apply H_w `chain` times, export: the inner
           loop of a hand-written filter or Lanczos on H_w (internal fields exist to be chained)
  apply    one call of `apply_Hw` / `apply_dslash` on canonical device buffers: a program that keeps
           its own layout and calls the operator once
  overlap  one call of `apply_overlap`: the overlap operator D(m) of a single source or of the 12
           spin-colour sources, with or without deflated low modes
  normal   one call of `apply_normal`: the operator D(m)^dag D(m) of a user's own solver, in the
           accurate arithmetic of a residual
  lowmodes `project_lowmodes` and `lowmode_update` on the tensor cores: the deflation of Eq. 7 alone
  cg       `cg_solve`: propagator columns to the FP64 true residual 1e-10
  net      `net_loss_grad`: forward and backward of the learned preconditioner on training pairs

The listed sizes are those of the repository's configurations, benchmark and tests: 4^4 (the plain
FP64 configuration), 8^4 and 8^3 x 16 (the propagators the benchmark and the tests solve),
16^3 x 32 (the deflated operator tests) and 24^3 x 64 (the dslash and overlap configurations).
`tune` marks the programs that call the autotuner once per lattice, as the benchmark does for its
large runs; the others take the library's default launch.

The sign polynomial's interval [eps, 1] reaches down to |lambda| = sqrt(eps) 6.6 < 0.47, below the gap
of H_w on these smoothed fields (0.5 at 24^3 x 64), so it holds the spectrum without deflation; the
deflated cases take away arbitrary directions.

Gauge fields: exp(i s H), H Gaussian in the Gell-Mann basis, then APE steps (alpha 0.6) and
re-unitarisation; antiperiodic time; Gaussian or point sources.
"""
import math

import numpy as np
import torch

from paper_1106_4964_gb300 import Context

BC = (1.0, 1.0, 1.0, -1.0)
RHO = 1.5
LMAX = 6.6  # above the free-field maximum of |H_w|, 8 - rho = 6.5


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # the smallest call: H_w once on the 4^4 lattice, where the launches are the cost
        case("hw_apply_f32_4c4", "apply", (4, 4, 4, 4), "f32", 1, s=0.3, ape=0, g5=1),
        # Wilson dslash throughput at the paper's precision, one source (the benchmark's headline)
        case("hw_f64_24c64", "hw", (24, 24, 24, 64), "f64", 1, chain=4, tune=1),
        # Wilson dslash throughput, the 12 sources of a propagator in one launch
        case("hw_f32_r12_24c64", "hw", (24, 24, 24, 64), "f32", 12, chain=8, tune=1),
        # a program with its own layout, a lattice that is no multiple of a block, 16-bit storage
        case("apply_bf16_r5_14x10x18x30", "apply", (14, 10, 18, 30), "bf16", 5),
        # the plain FP64 configuration: degree 100, 4^4, one Gaussian source
        case("overlap_f64_4c4", "overlap", (4, 4, 4, 4), "f64", 1, eps=0.005, degree=100),
        # one column of a propagator's operator with 100 deflated modes, order 200
        case("overlap_f32_nev100_16c32", "overlap", (16, 16, 16, 32), "f32", 1, eps=0.005, degree=200, nev=100,
             mass=0.02, tune=1),
        # the 16-bit form of the order-200 operator on the large lattice
        case("overlap_f16_24c64", "overlap", (24, 24, 24, 64), "f16", 1, eps=0.005, degree=200, tune=1),
        # true residuals of the 12 sources in double-float, on the benchmark's propagator lattice
        case("normal_df64_r12_8x16", "normal", (8, 8, 8, 16), "df64", 12, eps=0.005, degree=140, mass=0.05),
        # deflation of the 12 sources by 100 modes (Eq. 7) on the tensor cores
        case("lowmodes_f32_r12_16c32", "lowmodes", (16, 16, 16, 32), "f32", 12, nev=100),
        # the plain FP64 configuration's solve
        case("cg_f64_4c4", "cg", (4, 4, 4, 4), "f64", 1, eps=0.005, degree=100, mass=0.05),
        # a propagator: 12 point sources, FP32 inner operator in one chiral sector, FP64 true residuals
        case("cg_f32_r12_8c4", "cg", (8, 8, 8, 8), "f32", 12, eps=0.005, degree=150, mass=0.05, chiral=1, tune=1),
        # a training step's forward and backward over 8 recorded pairs
        case("net_grad_r8_8x16", "net", (8, 8, 8, 16), "f32", 8),
    ]


def case(name, kind, dims, prec, nrhs, s=0.5, ape=3, chain=1, g5=0, eps=0.0, degree=0, nev=0, mass=0.0, chiral=0,
         tune=0):
    return {"name": name, "kind": kind, "lx": dims[0], "ly": dims[1], "lz": dims[2], "lt": dims[3], "prec": prec,
            "nrhs": nrhs, "s": s, "ape": ape, "chain": chain, "g5": g5, "eps": eps, "degree": degree, "nev": nev,
            "mass": mass, "chiral": chiral, "tune": tune}


def draw(rng):
    """One more case of the same ranges: lattices between 4^4 and 24^3 x 64 whose volume is spread over
    its logarithm, any even extents, every storage precision, 1 to 12 sources."""
    c = _draw(rng)
    del c["name"]
    return c


def _draw(rng):
    kind = rng.choice(["hw", "hw", "apply", "apply", "overlap", "overlap", "overlap", "normal", "lowmodes", "cg",
                       "net"])
    top = {"hw": 24 ** 3 * 64, "apply": 24 ** 3 * 64, "overlap": 16 ** 3 * 32, "normal": 8 ** 3 * 16,
           "lowmodes": 16 ** 3 * 32, "cg": 8 ** 3 * 4, "net": 8 ** 3 * 16}[kind]
    lo = 4 ** 4 if kind != "lowmodes" else 4 ** 3 * 16
    vol = math.exp(rng.uniform(math.log(lo), math.log(top)))
    dims = _draw_dims(rng, vol, top)
    if kind in ("hw", "apply"):
        prec = rng.choice(["f64", "f32", "f32", "f16", "bf16", "df64"])
        nrhs = rng.choice([1, 1, 2, 3, 5, 7, 12]) if prec in ("f32", "f16", "bf16") else rng.choice([1, 1, 2, 3])
        chain = rng.randint(2, 8) if kind == "hw" else 1
        return case(None, kind, dims, prec, nrhs, chain=chain, g5=rng.randint(0, 1), tune=rng.randint(0, 1))
    if kind in ("overlap", "normal"):
        prec = rng.choice(["f64", "f32", "f32", "f16", "bf16", "df64"])
        big = dims[0] * dims[1] * dims[2] * dims[3] > 8 ** 3 * 16
        nrhs = rng.choice([1, 1, 2, 5, 12]) if prec in ("f32", "f16", "bf16") or not big else 1
        degree = rng.randint(20, 60) if prec in ("f64", "df64") and big else rng.randint(40, 200)
        nev = rng.choice([0, 0, rng.randint(1, 100)])
        return case(None, kind, dims, prec, nrhs, eps=round(rng.uniform(0.002, 0.005), 4), degree=degree, nev=nev,
                    mass=round(rng.uniform(0.0, 0.1), 3), tune=rng.randint(0, 1))
    if kind == "lowmodes":
        return case(None, kind, dims, rng.choice(["f32", "f32", "f16", "bf16"]), rng.choice([1, 3, 6, 12]),
                    nev=rng.randint(8, 128))
    if kind == "cg":
        inner = rng.choice(["f64", "f32", "f32"])
        if inner == "f64":
            dims = _draw_dims(rng, math.exp(rng.uniform(math.log(256), math.log(384))), 384)
        chiral = 0 if inner == "f64" else rng.randint(0, 1)
        nrhs = 12 if chiral else (1 if inner == "f64" else rng.choice([1, 3]))
        return case(None, kind, dims, inner, nrhs, eps=0.005,
                    degree=rng.randint(80, 100) if inner == "f64" else rng.randint(100, 150),
                    mass=round(rng.uniform(0.05, 0.15), 3), chiral=chiral)
    return case(None, kind, dims, "f32", rng.randint(1, 8))


def _draw_dims(rng, vol, top):
    """Even extents, the time extent the largest, with a volume near `vol` and at most `top`."""
    while True:
        e = vol ** 0.25
        d = [max(2, 2 * round(e * math.exp(rng.uniform(-0.35, 0.25)) / 2)) for _ in range(3)]
        t = max(2, 2 * round(vol / (d[0] * d[1] * d[2]) / 2))
        if min(d) >= 4 and 4 <= t <= 96 and 256 <= d[0] * d[1] * d[2] * t <= top:
            return (d[0], d[1], d[2], t)
        vol = min(top * 0.9, max(260.0, vol * math.exp(rng.uniform(-0.1, 0.1))))


# ------------------------------------------------------------------ inputs
def _dims(c):
    return (c["lx"], c["ly"], c["lz"], c["lt"])


def _gen(seed, what):
    g = torch.Generator(device="cuda")
    g.manual_seed(1000003 * (int(seed) + 1) + what)
    return g


def _gell_mann():
    m = torch.zeros(8, 3, 3, dtype=torch.complex128)
    m[0, 0, 1] = m[0, 1, 0] = 1
    m[1, 0, 1], m[1, 1, 0] = -1j, 1j
    m[2, 0, 0], m[2, 1, 1] = 1, -1
    m[3, 0, 2] = m[3, 2, 0] = 1
    m[4, 0, 2], m[4, 2, 0] = -1j, 1j
    m[5, 1, 2] = m[5, 2, 1] = 1
    m[6, 1, 2], m[6, 2, 1] = -1j, 1j
    m[7, 0, 0] = m[7, 1, 1] = 1 / math.sqrt(3)
    m[7, 2, 2] = -2 / math.sqrt(3)
    return m.cuda()


def _mul(a, b):
    """Product of 3x3 matrices held in the last two axes."""
    return sum(a[..., :, j:j + 1] * b[..., j:j + 1, :] for j in range(3))


def _su3(u):
    """Gram-Schmidt of rows 1 and 2, row 3 = conj(row1 x row2)."""
    r1 = u[..., 0, :]
    r1 = r1 / torch.linalg.vector_norm(r1, dim=-1, keepdim=True)
    r2 = u[..., 1, :]
    r2 = r2 - (r1.conj() * r2).sum(-1, keepdim=True) * r1
    r2 = r2 / torch.linalg.vector_norm(r2, dim=-1, keepdim=True)
    return torch.stack([r1, r2, torch.linalg.cross(r1, r2, dim=-1).conj()], dim=-2)


def _gauge(c, seed):
    """[Lt, Lz, Ly, Lx, 4, 3, 3] complex128 on the GPU."""
    lx, ly, lz, lt = _dims(c)
    h = torch.randn(lt, lz, ly, lx, 4, 8, generator=_gen(seed, 1), device="cuda", dtype=torch.float64)
    x = (0.5j * c["s"] / 32.0) * torch.einsum("...a,aij->...ij", h.to(torch.complex128), _gell_mann())
    eye = torch.eye(3, dtype=torch.complex128, device="cuda")
    u = eye + x / 8.0
    for j in range(7, 0, -1):  # exp of 1/32 of the exponent by an 8-term series, then five squarings
        u = eye + _mul(x, u) / j
    for _ in range(5):
        u = _mul(u, u)
    u = _su3(u)
    axis = (3, 2, 1, 0)
    for _ in range(c["ape"]):
        out = []
        for mu in range(4):
            um = u[..., mu, :, :]
            st = torch.zeros_like(um)
            for nu in range(4):
                if nu == mu:
                    continue
                un = u[..., nu, :, :]
                st += _mul(_mul(un, torch.roll(um, -1, axis[nu])), torch.roll(un, -1, axis[mu]).mH)
                ub = torch.roll(un, 1, axis[nu])
                st += _mul(_mul(ub.mH, torch.roll(um, 1, axis[nu])), torch.roll(ub, -1, axis[mu]))
            out.append(_su3(0.4 * um + 0.1 * st))
        u = torch.stack(out, dim=-3)
    return u.contiguous()


def _spinor(c, seed, what, nrhs):
    lx, ly, lz, lt = _dims(c)
    return torch.randn(nrhs, lt, lz, ly, lx, 4, 3, generator=_gen(seed, what), device="cuda", dtype=torch.complex128)


def _source(c, seed):
    """Gaussian sources, or the spin-colour point sources of a propagator at a random site."""
    if c["kind"] == "cg" and c["nrhs"] == 12:
        lx, ly, lz, lt = _dims(c)
        n = int(torch.randint(lx * ly * lz * lt, (1,), generator=_gen(seed, 7), device="cuda").item())
        b = torch.zeros(12, lx * ly * lz * lt, 12, dtype=torch.complex128, device="cuda")
        b[torch.arange(12), n, torch.arange(12)] = 1.0
        return b.view(12, lt, lz, ly, lx, 4, 3)
    return _spinor(c, seed, 2, c["nrhs"])


def _modes(c, seed):
    """nev orthonormal fields and signed values: Eq. 7 is a formula in any orthonormal set, so seeded
    ones stand in for the modes an eigensolver takes minutes to find."""
    n = c["nev"]
    v = _spinor(c, seed, 3, n).view(n, -1)
    for _ in range(2):
        g = v.conj() @ v.T
        low = torch.linalg.cholesky(g)
        v = torch.linalg.solve_triangular(low.conj(), v, upper=False)
    vals = torch.rand(n, 2, generator=_gen(seed, 4), device="cuda", dtype=torch.float64).cpu().numpy()
    return np.where(vals[:, 1] < 0.5, -1.0, 1.0) * (0.05 + 0.35 * vals[:, 0]), v.contiguous()


def _net_weights(seed):
    w = torch.randn(2, 9 * 16 * 16, generator=_gen(seed, 5), device="cuda", dtype=torch.complex128)
    return 0.2 * w.view(2, 9 * 16, 4, 4)


def prepare(case, seed):
    c = case
    ctx = Context(_dims(c), BC)
    ctx.set_gauge(_gauge(c, seed))
    st = {"case": c, "ctx": ctx}
    if c["tune"]:
        ctx.tune_dslash(_work_prec(c), c["nrhs"])
    if c["degree"]:
        ctx.set_sign_poly(RHO, c["eps"], c["degree"], LMAX)
    if c["nev"]:
        vals, vecs = _modes(c, seed)
        ctx.set_eigenpairs(0, vals, vecs)
        del vecs
    if c["kind"] == "net":
        ctx.net_set_weights(_net_weights(seed).cpu().numpy().reshape(-1))
        st["e"] = _spinor(c, seed, 6, c["nrhs"])
    st["x"] = _source(c, seed)
    if c["kind"] in ("hw", "lowmodes"):
        st["f"] = [ctx.field(c["nrhs"], c["prec"]) for _ in range(3)]
    if c["kind"] == "cg":
        ctx.set_option("chiral", c["chiral"])
    st["out"] = torch.empty_like(st["x"])
    if c["kind"] == "lowmodes":
        st["out2"] = torch.empty_like(st["x"])
    return st


def _work_prec(c):
    """The storage the operator's launches run in: 16-bit overlap keeps FP32 recurrence vectors."""
    return "f32" if c["kind"] in ("overlap", "normal") and c["prec"] in ("f16", "bf16") else c["prec"]


# ------------------------------------------------------------------ one pass
def run(state):
    c, ctx, x, out = state["case"], state["ctx"], state["x"], state["out"]
    kind = c["kind"]
    if kind == "apply":
        (ctx.apply_Hw if c["g5"] else ctx.apply_dslash)(x, out, -RHO, prec=c["prec"])
        return out
    if kind == "hw":
        f = state["f"]
        f[0].load(x)
        for k in range(c["chain"]):
            ctx.dslash_field(f[k & 1], f[1 - (k & 1)], -RHO, gamma5=True)
        f[c["chain"] & 1].store(out)
        return out
    if kind == "overlap":
        ctx.apply_overlap(x, out, c["mass"], prec=c["prec"])
        return out
    if kind == "normal":
        ctx.apply_normal(x, out, c["mass"], prec=c["prec"])
        return out
    if kind == "lowmodes":
        f = state["f"]
        f[0].load(x)
        coef = ctx.project_lowmodes(0, f[0], engine=2 if c["prec"] == "f32" else 1)
        ctx.lowmode_update(0, f[0], coef, f[1], f[2], engine=1)
        f[1].store(out)
        f[2].store(state["out2"])
        return {"coef": coef, "high": out, "low": state["out2"]}
    if kind == "cg":
        ctx.cg_solve(x, out, mass=c["mass"], tol=1e-10, max_iter=2000, inner_prec=c["prec"])
        return out
    loss, grad = ctx.net_loss_grad(x, state["e"])
    return {"loss": loss, "grad": grad}


# ------------------------------------------------------------------ what it takes
_REAL = {"f64": 8, "f32": 4, "f16": 2, "bf16": 2, "df64": 8}


def work(case):
    """Links as their first two rows (16 complex numbers would be redundant), fields in their storage
    precision, canonical buffers in complex128; 1320 flop per site and D_w."""
    c = case
    V, R, rb = math.prod(_dims(c)), c["nrhs"], _REAL[c["prec"]]
    links = 48 * rb * V
    canon = 2 * 192 * V * R
    modes = 24 * (4 if rb == 2 else rb) * V * c["nev"]
    dw = 1320 * V * R
    proj = 96 * V * R * c["nev"]
    kind = c["kind"]
    if kind == "apply":
        return {"bytes": links + canon, "flops": dw}
    if kind == "hw":
        return {"bytes": canon + c["chain"] * (links + 48 * rb * V * R), "flops": c["chain"] * dw}
    if kind == "overlap":
        return {"bytes": links + canon + modes, "flops": (2 * c["degree"] + 1) * dw + 3 * proj}
    if kind == "normal":
        return {"bytes": links + canon + modes, "flops": 2 * (2 * c["degree"] + 1) * dw + 6 * proj}
    if kind == "lowmodes":
        return {"bytes": 3 * 192 * V * R + modes, "flops": 3 * proj}
    if kind == "cg":
        # a solve of these masses takes about 40 iterations, one or two sign applications each
        it = 40 * (1 if c["chiral"] else 2)
        return {"bytes": links + canon, "flops": it * (2 * c["degree"] + 1) * dw}
    # forward, input gradient and weight gradients of two layers of 9 paths x 16 channels: a spin mix of
    # 16 x 3 complex products each, and one transport of a spinor per path and layer
    return {"bytes": links + canon, "flops": R * V * (4 * 9 * 16 * 48 * 8 + 3 * 9 * 4 * 66)}


# ------------------------------------------------------------------ tolerances
def tolerance(case):
    """About four times the distance from exact() that the path shows over these ranges."""
    c = case
    p, kind = c["prec"], c["kind"]
    if kind == "cg":
        # a residual of 1e-10 leaves an error of up to cond(D^dag D) ~ (2 rho / m)^2 times that
        return {"rel": 2e-8}
    if kind == "net":
        return {"rel": 5e-7}
    if kind in ("apply", "hw"):
        return {"rel": {"f64": 1e-15, "df64": 2e-14, "f32": 4e-7, "f16": 1.5e-3, "bf16": 1e-2}[p]}
    if kind == "lowmodes":
        return {"rel": {"f32": 5e-5, "f16": 1e-2, "bf16": 1e-2}[p]}
    return {"rel": {"f64": 1e-13, "df64": 2e-13, "f32": 1.5e-6, "f16": 1.5e-3, "bf16": 1e-2}[p]}


# ------------------------------------------------------------------ the same in 64 bits, plain torch
_AX = (-3, -4, -5, -6)  # axis of direction mu in [..., t, z, y, x, spin, colour]


def _hop(x, u, mu, fwd):
    """T x(n) = U_mu(n) x(n + mu) or U_mu(n - mu)^dag x(n - mu), with the boundary phase; any spins."""
    if fwd:
        y = torch.roll(x, -1, _AX[mu])
        if BC[mu] != 1.0:
            y.select(_AX[mu], y.shape[_AX[mu]] - 1).mul_(BC[mu])
        w = u[..., mu, :, :].unsqueeze(-3)  # [t, z, y, x, 1, i, j]
        return sum(w[..., :, j] * y[..., j:j + 1] for j in range(3))
    w = u[..., mu, :, :].unsqueeze(-3).conj()
    y = torch.roll(sum(w[..., j, :] * x[..., j:j + 1] for j in range(3)), 1, _AX[mu])
    if BC[mu] != 1.0:
        y.select(_AX[mu], 0).mul_(BC[mu])
    return y


def _amul(mu, d, dag):
    """A_mu d (or A_mu^dag d) on two spins; gamma_mu = [[0, A_mu], [A_mu^dag, 0]], A_k = -i sigma_k, A_4 = 1."""
    a, b = d[..., 0, :], d[..., 1, :]
    g = 1.0 if dag else -1.0
    if mu == 0:
        return torch.stack([1j * g * b, 1j * g * a], dim=-2)
    if mu == 1:
        return torch.stack([g * b, -g * a], dim=-2)
    if mu == 2:
        return torch.stack([1j * g * a, -1j * g * b], dim=-2)
    return d


def _dslash(x, u, m, g5=False):
    out = (4.0 + m) * x
    for mu in range(4):
        for fwd in (True, False):
            sg = 1.0 if fwd else -1.0
            h = x[..., :2, :] - sg * _amul(mu, x[..., 2:, :], False)
            h = _hop(h, u, mu, fwd)
            out[..., :2, :] -= 0.5 * h
            out[..., 2:, :] += 0.5 * sg * _amul(mu, h, True)
    if g5:
        out[..., 2:, :] *= -1.0
    return out


def _cheb(eps, n):
    m = n + 1
    th = math.pi * (np.arange(m) + 0.5) / m
    f = 1.0 / np.sqrt(0.5 * (1.0 + eps) + 0.5 * (1.0 - eps) * np.cos(th))
    c = 2.0 / m * np.cos(np.outer(np.arange(m), th)) @ f
    c[0] *= 0.5
    return c


def _overlap(x, u, c, vals, vecs, mass):
    """D(m) x: the low modes exactly, P(Q^2) of the rest by Clenshaw's recurrence."""
    shape = x.shape
    low = torch.zeros_like(x)
    psi = x
    if vecs is not None:
        k = vecs.conj() @ x.reshape(shape[0], -1).T
        psi = (x.reshape(shape[0], -1) - (vecs.T @ k).T).view(shape)
        low = (vecs.T @ (torch.sign(vals)[:, None] * k)).T.reshape(shape)
    cf = _cheb(c["eps"], c["degree"])
    e = c["eps"]
    b1, b2 = torch.zeros_like(x), torch.zeros_like(x)
    for k in range(c["degree"], -1, -1):
        q2 = _dslash(_dslash(b1, u, -RHO, True), u, -RHO, True) / LMAX ** 2
        y = (2.0 * q2 - (1.0 + e) * b1) / (1.0 - e)
        b1, b2 = cf[k] * psi + (2.0 if k else 1.0) * y - b2, b1
    sign = low + _dslash(b1, u, -RHO, True) / LMAX
    sign[..., 2:, :] *= -1.0
    return (RHO + 0.5 * mass) * x + (RHO - 0.5 * mass) * sign


def _normal(x, u, c, vals, vecs, mass):
    y = _overlap(x, u, c, vals, vecs, mass)
    y[..., 2:, :] *= -1.0
    y = _overlap(y, u, c, vals, vecs, mass)
    y[..., 2:, :] *= -1.0
    return y


def _solve(b, u, c):
    """D(m)^dag D(m) x = b on a small lattice from the dense H_w and its eigenvectors."""
    n = b[0].numel()
    eye = torch.eye(n, dtype=torch.complex128, device="cuda").view(n, *b.shape[1:])
    h = torch.empty(n, n, dtype=torch.complex128, device="cuda")
    for i in range(0, n, 256):
        h[:, i:i + 256] = _dslash(eye[i:i + 256], u, -RHO, True).reshape(-1, n).T
    lam, v = torch.linalg.eigh(0.5 * (h + h.mH))
    q2 = (lam / LMAX) ** 2
    y = (2.0 * q2 - (1.0 + c["eps"])) / (1.0 - c["eps"])
    p = torch.from_numpy(np.polynomial.chebyshev.chebval(y.cpu().numpy(), _cheb(c["eps"], c["degree"]))).cuda()
    d = (v * (lam / LMAX * p)) @ v.mH
    g5 = torch.ones(b.shape[1:], dtype=torch.float64, device="cuda")
    g5[..., 2:, :] = -1.0
    d = (RHO - 0.5 * c["mass"]) * g5.reshape(-1, 1) * d
    d.diagonal().add_(RHO + 0.5 * c["mass"])
    x = b.reshape(b.shape[0], -1).T
    return torch.linalg.solve(d, torch.linalg.solve(d.mH, x)).T.reshape(b.shape)


def _net(u, w, r, e):
    """loss = sum_k |M r_k - e_k|^2 / |e_k|^2 and d/dRe W + i d/dIm W, M = L2 L1."""
    w1 = w[0].view(9, 16, 4, 4).clone().requires_grad_(True)
    w2 = w[1].view(9, 16, 4, 4).clone().requires_grad_(True)

    def paths(x):
        return [x] + [_hop(x, u, mu, f) for mu in range(4) for f in (True, False)]

    loss = 0.0
    for k in range(r.shape[0]):
        t1 = torch.stack(paths(r[k]))
        h = torch.einsum("pcst,p...ti->c...si", w1, t1)
        y = sum(torch.einsum("cst,c...ti->...si", w2[p], t) for p, t in enumerate(paths(h)))
        d = y - e[k]
        loss = loss + (d.real ** 2 + d.imag ** 2).sum() / (e[k].real ** 2 + e[k].imag ** 2).sum()
    loss.backward()
    return {"loss": float(loss.item()),
            "grad": torch.cat([w1.grad.reshape(-1), w2.grad.reshape(-1)]).cpu().numpy()}


def exact(case, seed):
    c = case
    V, R = math.prod(_dims(c)), c["nrhs"]
    u = _gauge(c, seed)
    x = _source(c, seed)
    kind = c["kind"]
    if kind in ("apply", "hw"):
        for _ in range(c["chain"]):
            x = _dslash(x, u, -RHO, kind == "hw" or bool(c["g5"]))
        return x
    if kind == "cg":
        return _solve(x, u, c) if V <= 320 else None
    if kind == "net":
        return _net(u, _net_weights(seed), x, _spinor(c, seed, 6, R))
    vals = vecs = None
    if c["nev"]:
        vals, vecs = _modes(c, seed)
        vals = torch.from_numpy(vals).cuda().to(torch.complex128)
    if kind == "lowmodes":
        flat = x.reshape(R, -1)
        k = vecs.conj() @ flat.T
        low = (vecs.T @ (torch.sign(vals.real)[:, None] * k)).T.reshape(x.shape).clone()
        low[..., 2:, :] *= -1.0
        return {"coef": k.cpu().numpy(), "high": (flat - (vecs.T @ k).T).view(x.shape), "low": low}
    if vals is not None:
        vals = vals.real
    # about 100 small launches a D_w in plain torch, or their memory traffic
    per = max(8e-4, 2.5e-9 * 4 * V * R)
    if per * 2 * c["degree"] * (2 if kind == "normal" else 1) > 20.0:
        return None
    f = _overlap if kind == "overlap" else _normal
    return f(x, u, c, vals, vecs, c["mass"])
