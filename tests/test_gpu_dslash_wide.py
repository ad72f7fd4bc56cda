"""The FP64 and double-float dslash at the edges of its fixed-point hop: fields whose neighbouring
sites differ by many orders of magnitude, vanishing neighbours and components, infinities and NaN,
scales near the ends of the exponent range, and every launch variant on ragged site groups."""
import numpy as np
import pytest

import oracle
import synth
from gpu_common import ABC, RHO, TOL, dev, host, need_gpu, rel, torch

pytestmark = pytest.mark.gpu

DIMS = (6, 4, 4, 6)


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    need_gpu()


def apply(prec, U, psi, dims=DIMS):
    from paper_1106_4964_gb300 import Context

    ctx = Context(dims, ABC)
    ctx.set_gauge(dev(U))
    out = torch.empty_like(dev(psi))
    ctx.apply_dslash(dev(psi), out, -RHO, prec=prec)
    return host(out)


def fields():
    rng = np.random.default_rng(7)
    base = synth.gaussian_spinor(DIMS, 2)
    site = 2.0 ** rng.integers(-40, 41, base.shape[:5])[..., None, None]
    comp = 2.0 ** rng.integers(-35, 36, base.shape)
    colour0 = base.copy()
    colour0[..., 1:] = 0  # zero components in every neighbour
    sector = base.copy()
    sector[..., 2:, :] = 0
    return {"site_scales": base * site, "component_scales": base * comp, "one_colour": colour0,
            "one_chirality": sector, "point": synth.point_sources(DIMS)[4:5], "zero": np.zeros_like(base)}


@pytest.mark.parametrize("name", sorted(fields()))
@pytest.mark.parametrize("prec", ["f64", "df64"])
def test_uneven_fields(prec, name):
    """Site by site: the error relative to the largest of the nine spinors a site reads."""
    U = synth.gauge_field(DIMS, 1, 0.5)
    psi = fields()[name]
    got = apply(prec, U, psi)[0]
    ref = oracle.dslash(DIMS, ABC, U, -RHO, psi).reshape(got.shape)
    mag = np.abs(psi[0]).max(axis=(-2, -1))
    near = mag.copy()
    for ax in range(4):
        near = np.maximum(near, np.maximum(np.roll(mag, 1, ax), np.roll(mag, -1, ax)))
    err = np.abs(got - ref).max(axis=(-2, -1))
    assert np.all(err <= TOL[prec] * near)
    if name == "zero":
        assert not got.any()


@pytest.mark.parametrize("prec,scale", [("f64", 1e-290), ("f64", 1e-200), ("f64", 1e290), ("df64", 1e-20), ("df64", 1e30)])
def test_scales(prec, scale):
    U = synth.gauge_field(DIMS, 1, 0.5)
    psi = synth.gaussian_spinor(DIMS, 2)
    got = apply(prec, U, psi * scale) / scale
    assert rel(got, oracle.dslash(DIMS, ABC, U, -RHO, psi)) <= TOL[prec]


@pytest.mark.parametrize("prec", ["f64", "df64"])
@pytest.mark.parametrize("value", [np.inf, np.nan])
def test_non_finite(prec, value):
    """One non-finite component: its site and the eight neighbours get non-finite components, every
    other site its value."""
    U = synth.gauge_field(DIMS, 1, 0.5)
    psi = synth.gaussian_spinor(DIMS, 2)
    ref = oracle.dslash(DIMS, ABC, U, -RHO, psi).reshape(psi.shape)[0]
    psi[0, 2, 1, 3, 4, 1, 2] = value
    got = apply(prec, U, psi)[0]
    bad = ~np.isfinite(got).all(axis=(-2, -1))
    want = np.zeros_like(bad)
    want[2, 1, 3, 4] = True
    for ax in range(4):
        for st in (1, -1):
            want |= np.roll((np.indices(want.shape) == np.array([2, 1, 3, 4]).reshape(4, 1, 1, 1, 1)).all(0), st, ax)
    assert np.array_equal(bad, want)
    assert rel(got[~bad], ref[~bad]) <= TOL[prec]


@pytest.mark.parametrize("shape", [(32, 1, 0), (32, 3, 1), (64, 2, 2), (256, 1, 1)])
@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (2, 6, 4, 10), (6, 4, 4, 6)])
@pytest.mark.parametrize("prec", ["f64", "df64"])
def test_launch_shapes(prec, dims, shape):
    from paper_1106_4964_gb300 import Context

    U = synth.gauge_field(dims, 5, 0.5)
    psi = synth.gaussian_spinor(dims, 6, nrhs=4)
    ctx = Context(dims, ABC)
    ctx.set_gauge(dev(U))
    ctx.set_dslash_shape(prec, 4, *shape)
    out = torch.empty_like(dev(psi))
    ctx.apply_dslash(dev(psi), out, -RHO, prec=prec)
    got = host(out)
    for r in range(4):
        assert rel(got[r], oracle.dslash(dims, ABC, U, -RHO, psi[r])) <= TOL[prec]


@pytest.mark.parametrize("nrhs", [3, 12])
@pytest.mark.parametrize("prec", ["f64", "df64"])
def test_autotuner_candidates(prec, nrhs):
    """Every candidate the autotuner times for several right-hand sides is a launch the library takes."""
    from paper_1106_4964_gb300 import Context

    U = synth.gauge_field(DIMS, 5, 0.5)
    psi = synth.gaussian_spinor(DIMS, 6, nrhs=nrhs)
    ctx = Context(DIMS, ABC)
    ctx.set_gauge(dev(U))
    shape = ctx.tune_dslash(prec, nrhs)
    ctx.set_dslash_shape(prec, nrhs, *shape)
    out = torch.empty_like(dev(psi))
    ctx.apply_dslash(dev(psi), out, -RHO, prec=prec)
    got = host(out)
    for r in range(nrhs):
        assert rel(got[r], oracle.dslash(DIMS, ABC, U, -RHO, psi[r])) <= TOL[prec]


@pytest.mark.parametrize("prec", ["f64", "df64"])
def test_phase_next_to_one(prec):
    """A real boundary phase that FP32 rounds to 1 is applied."""
    from paper_1106_4964_gb300 import Context

    bc = (1.0, 1.0 - 2.0 ** -27, 1.0, 1.0 + 2.0 ** -25)
    U = synth.gauge_field(DIMS, 1, 0.5)
    psi = synth.gaussian_spinor(DIMS, 2)
    ctx = Context(DIMS, bc)
    ctx.set_gauge(dev(U))
    out = torch.empty_like(dev(psi))
    ctx.apply_dslash(dev(psi), out, -RHO, prec=prec)
    ref = oracle.dslash(DIMS, bc, U, -RHO, psi[0])
    assert rel(oracle.dslash(DIMS, (1.0,) * 4, U, -RHO, psi[0]), ref) > 100 * TOL[prec]
    assert rel(host(out), ref) <= TOL[prec]


def diagonal_links(dims, seed):
    """SU(3) links that mix no colours: diag(e^ia, e^ib, e^-i(a+b))."""
    rng = np.random.default_rng(seed)
    a = rng.uniform(-3, 3, tuple(reversed(dims)) + (4, 2))
    U = np.zeros(a.shape[:-1] + (3, 3), dtype=np.complex128)
    for i, ph in enumerate((a[..., 0], a[..., 1], -a.sum(-1))):
        U[..., i, i] = np.exp(1j * ph)
    return U


@pytest.mark.parametrize("unit", [True, False])
@pytest.mark.parametrize("prec", ["f64", "df64"])
def test_empty_colours_stay_empty(prec, unit):
    """Links that mix no colours, sources in one colour: the others are exactly zero after any number of
    applications, as with floating-point arithmetic."""
    from paper_1106_4964_gb300 import Context

    U = diagonal_links(DIMS, 3)
    if unit:
        U[:] = np.eye(3)
    psi = synth.gaussian_spinor(DIMS, 2, nrhs=2)
    psi[0][..., [0, 2]] = 0
    psi[1] = 0
    psi[1, 0, 0, 0, 0, 2, 1] = 1  # a point source
    ctx = Context(DIMS, ABC)
    ctx.set_gauge(dev(U))
    f = [ctx.field(2, prec) for _ in range(2)]
    f[0].load(dev(psi))
    out = torch.empty_like(dev(psi))
    ref = psi.copy()
    for k in range(6):
        ctx.dslash_field(f[k & 1], f[1 - (k & 1)], -RHO)
        f[1 - (k & 1)].store(out)
        got = host(out)
        assert not got[..., [0, 2]].any()
        for r in range(2):
            ref[r] = oracle.dslash(DIMS, ABC, U, -RHO, ref[r]).reshape(ref[r].shape)
            assert rel(got[r], ref[r]) <= TOL[prec]
    for a in f:
        a.close()


def reference(dims, bc, U, m, psi):
    """D_w psi in extended precision, and the weight of its roundings: |4 + m| |psi| + 1/2 sum |U_ij| |h_j|."""
    U, psi = U.astype(np.clongdouble), psi.astype(np.clongdouble)
    up, dn = psi[..., :2, :], psi[..., 2:, :]
    out, w = (4 + np.longdouble(m)) * psi, abs(4 + m) * np.abs(psi)

    def amul(mu, d, g):  # A_mu d (g = -1) or A_mu^dag d (g = 1)
        a, b = d[..., 0, :], d[..., 1, :]
        x = [(1j * g * b, 1j * g * a), (g * b, -g * a), (1j * g * a, -1j * g * b), (a, b)][mu]
        return np.stack(x, axis=-2)

    for mu in range(4):
        ax = 3 - mu
        for s in (1, -1):
            h = up - s * amul(mu, dn, -1)
            u = U[..., mu, :, :]
            edge = [slice(None)] * 6
            edge[ax] = -1 if s > 0 else 0
            if s > 0:
                h = np.roll(h, -1, ax)
            else:
                u = np.conj(np.swapaxes(u, -1, -2))
            chi, mag = np.einsum("...ij,...aj->...ai", u, h), np.einsum("...ij,...aj->...ai", np.abs(u), np.abs(h))
            if s < 0:
                chi, mag = np.roll(chi, 1, ax), np.roll(mag, 1, ax)
            chi[tuple(edge)] *= bc[mu]
            out[..., :2, :] -= chi / 2
            out[..., 2:, :] += s * amul(mu, chi, 1) / 2
            w[..., :2, :] += mag / 2
            w[..., 2:, :] += mag[..., ::-1, :] / 2 if mu < 2 else mag / 2
    return out, w


def component_cases():
    rng = np.random.default_rng(11)
    base = synth.gaussian_spinor(DIMS, 2)
    mixing, diag = synth.gauge_field(DIMS, 1, 0.5), diagonal_links(DIMS, 3)
    weak = synth.gauge_field(DIMS, 1, 1e-9)  # off-diagonal entries of 1e-9: below the fixed-point links' last bits
    colours = base * 2.0 ** np.array([0.0, -30.0, -50.0])
    spread = base * 2.0 ** rng.integers(-35, 36, base.shape)
    site = base * 2.0 ** rng.integers(-40, 41, base.shape[:5])[..., None, None]
    one = base.copy()
    one[..., 1:] = 0
    near = base * 2.0 ** -rng.integers(0, 12, base.shape)  # across the line below which a component is formed again
    return {"mixing": (mixing, base), "mixing_spread": (mixing, spread), "mixing_site": (mixing, site),
            "mixing_near": (mixing, near), "diagonal_colours": (diag, colours), "diagonal_spread": (diag, spread),
            "diagonal_site": (diag, site), "diagonal_near": (diag, near), "weak_one_colour": (weak, one),
            "weak_colours": (weak, colours), "point": (diag, synth.point_sources(DIMS)[4:5])}


@pytest.mark.parametrize("name", sorted(component_cases()))
@pytest.mark.parametrize("prec", ["f64", "df64"])
def test_every_component_keeps_its_precision(prec, name):
    """Component by component against extended precision.  Floating point: 24 roundings of the products and
    sums that make a component, and 4 of the epilogue.  Fixed point: 8 hops of at most 3.6 units of 2^-58 of the
    scale, 2^6 (FP64) or 2^9 (double-float) times which the component is: 2^-47.1 or 2^-44.1 of it.  Both are
    below 64 units of 2^-53 (FP64) or 2^-47 (double-float: 24 operations of 2^-46)."""
    U, psi = component_cases()[name]
    if prec == "df64":  # the pair's 48 bits
        hi = psi.view(np.float64).astype(np.float32)
        psi = (hi.astype(np.float64) + (psi.view(np.float64) - hi).astype(np.float32)).view(np.complex128)
    got = apply(prec, U, psi)[0]
    ref, w = reference(DIMS, ABC, U, -RHO, psi[0])
    err = np.abs(got.astype(np.clongdouble) - ref).astype(np.float64)
    bound = 64 * {"f64": 2.0 ** -53, "df64": 2.0 ** -47}[prec] * w.astype(np.float64)
    worst = float((err / np.where(bound > 0, bound, 1)).max())
    print(f"{prec} {name}: {worst:.2e} of the bound")
    assert np.all(err <= bound), worst


@pytest.mark.parametrize("prec,tol", [("f64", 6e-16), ("double_float", 5e-15)])
def test_roundings_do_not_add_up(prec, tol):
    """Twelve applications against extended precision: an unbiased rounding grows with the root of their number
    (2.5e-15 and 1.5e-16 for one, mostly the pair's and FP64's rounding of the result, of which D_w averages
    nine), a sum that is always cut short with the number itself (2.6e-15 each in double-float)."""
    from paper_1106_4964_gb300 import Context

    prec = {"double_float": "df64"}.get(prec, prec)
    U, psi = synth.gauge_field(DIMS, 1, 0.5), synth.gaussian_spinor(DIMS, 2)
    ctx = Context(DIMS, ABC)
    ctx.set_gauge(dev(U))
    f = [ctx.field(1, prec) for _ in range(2)]
    f[0].load(dev(psi))
    ref = psi[0].astype(np.clongdouble)
    for k in range(12):
        ctx.dslash_field(f[k & 1], f[1 - (k & 1)], -RHO)
        ref = reference(DIMS, ABC, U, -RHO, ref)[0]
    out = torch.empty_like(dev(psi))
    f[0].store(out)
    err = float(np.linalg.norm((host(out)[0] - ref).ravel()) / np.linalg.norm(ref.ravel()))
    print(f"{prec}: {err:.2e}")
    for a in f:
        a.close()
    assert err <= tol
