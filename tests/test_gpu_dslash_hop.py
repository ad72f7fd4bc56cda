"""The one-warp-per-hop launch of the FP32-arithmetic dslash (variant 12, the default on small lattices)
against the oracle: ragged site groups, several right-hand sides, gamma5 and the fused Clenshaw epilogue
with FP32 and 16-bit links, and the default launch on either side of its size limit."""
import numpy as np
import pytest

import oracle
import synth
from gpu_common import ABC, RHO, TOL, dev, host, need_gpu, rel, torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    need_gpu()


@pytest.mark.parametrize("dims,nrhs", [((2, 2, 2, 2), 1), ((2, 6, 4, 10), 3), ((6, 4, 4, 6), 2), ((34, 2, 2, 4), 1)])
@pytest.mark.parametrize("prec", ["f32", "f16", "bf16"])
def test_hop_variant(dims, nrhs, prec):
    from paper_1106_4964_gb300 import Context

    U = synth.gauge_field(dims, 5, 0.5)
    psi = synth.gaussian_spinor(dims, 6, nrhs=nrhs)
    ctx = Context(dims, ABC)
    ctx.set_gauge(dev(U))
    ctx.set_dslash_shape(prec, nrhs, 32, 1, 12)
    ctx.set_dslash_shape("f32", nrhs, 32, 1, 12)  # the 16-bit overlap's recurrence fields
    out = torch.empty_like(dev(psi))
    ctx.apply_Hw(dev(psi), out, -RHO, prec=prec)
    got = host(out)
    for r in range(nrhs):
        assert rel(got[r], oracle.hw(dims, ABC, U, -RHO, psi[r])) <= TOL[prec]
    eps, n, lmax = 0.05, 20, 9.0
    ctx.set_sign_poly(RHO, eps, n, lmax)
    ctx.apply_overlap(dev(psi), out, 0.02, prec=prec)
    got = host(out)
    c = oracle.cheb_coeffs(eps, n)
    for r in range(nrhs):
        assert rel(got[r], oracle.overlap(dims, ABC, U, RHO, 0.02, lmax, eps, c, psi[r])) <= TOL[prec]


@pytest.mark.parametrize("prec", ["f32", "f16", "bf16", "f64", "df64"])
# sites x sources on either side of the limits: 9000 (16-bit) and 13 000 (FP32), 12 000 (FP64, double-float), 50 000
@pytest.mark.parametrize("dims,nrhs", [((6, 6, 6, 10), 4), ((6, 6, 6, 10), 5), ((6, 6, 6, 10), 7), ((8, 8, 8, 8), 4),
                                       ((8, 8, 8, 8), 13), ((16, 8, 8, 16), 1), ((16, 8, 8, 16), 2)])
def test_default_launch(dims, nrhs, prec):
    from paper_1106_4964_gb300 import Context

    U = synth.gauge_field(dims, 5, 0.5)
    psi = synth.gaussian_spinor(dims, 6, nrhs=nrhs)
    ctx = Context(dims, ABC)
    ctx.set_gauge(dev(U))
    out = torch.empty_like(dev(psi))
    ctx.apply_dslash(dev(psi), out, -RHO, prec=prec)
    got = host(out)
    for r in range(nrhs):
        assert rel(got[r], oracle.dslash(dims, ABC, U, -RHO, psi[r])) <= TOL[prec]
