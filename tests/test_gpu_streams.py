"""Stream behaviour of the calls: a host buffer belongs to its caller again when the call returns."""
import pytest

import synth
from gpu_common import ABC, RHO, dev, host, need_gpu, torch

pytestmark = pytest.mark.gpu

DIMS = (8, 8, 8, 8)


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    need_gpu()


@pytest.fixture(scope="module")
def busy():
    """Work of some 20 ms on the current stream: what a call enqueues behind it has not begun when the call's
    host code ends."""
    a = torch.randn(8192, 8192, device="cuda")
    b = torch.empty_like(a)

    def go(n=2):
        for _ in range(n):
            torch.matmul(a, a, out=b)

    go()
    torch.cuda.synchronize()
    return go


def make():
    from paper_1106_4964_gb300 import Context

    ctx = Context(DIMS, ABC)
    ctx.set_gauge(dev(synth.gauge_field(DIMS, 5, 0.5)))
    ctx.set_sign_poly(RHO, 0.05, 20, 9.0)
    w = torch.randn(4608, dtype=torch.complex128, generator=torch.Generator().manual_seed(1))
    ctx.net_set_weights(0.1 * w.numpy())
    return ctx


CALLS = {
    "Hw": lambda ctx, x, out: ctx.apply_Hw(x, out, -RHO, prec="f32"),
    "overlap": lambda ctx, x, out: ctx.apply_overlap(x, out, 0.1, prec="f32"),
    "normal": lambda ctx, x, out: ctx.apply_normal(x, out, 0.1, prec="f64"),
    "net": lambda ctx, x, out: ctx.net_apply(x, out),
}


@pytest.mark.parametrize("name", ["Hw", "overlap", "normal", "net", "load"])
def test_host_input_may_be_reused(name, busy):
    """Pinned input, device output: overwriting the input after the call changes nothing."""
    ctx = make()
    psi = torch.from_numpy(synth.gaussian_spinor(DIMS, 6, nrhs=2))
    x, out = psi.clone().pin_memory(), torch.empty_like(dev(psi.numpy()))
    ref = torch.empty_like(out)
    if name == "load":
        f = ctx.field(2, "f64")
        f.load(x)  # warm: the staging buffer exists
        torch.cuda.synchronize()
        busy()
        f.load(x)
        x.zero_()
        f.store(out)
        assert torch.equal(out, psi.cuda())
        f.close()
        return
    CALLS[name](ctx, dev(psi.numpy()), ref)
    CALLS[name](ctx, x, out)
    torch.cuda.synchronize()
    out.zero_()
    busy()
    CALLS[name](ctx, x, out)
    x.zero_()
    assert (host(out) == host(ref)).all()
