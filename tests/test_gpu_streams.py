"""Stream behaviour of the calls: a host buffer belongs to its caller again when the call returns, and the
calls of one context, which share its work fields, take turns across streams."""
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


@pytest.mark.parametrize("second", ["null", "other"])
@pytest.mark.parametrize("name", ["Hw", "overlap", "normal", "net"])
def test_calls_on_two_streams_take_turns(name, second, busy):
    """The first call sits behind other work of its stream when the second, on an idle stream, is made."""
    ctx = make()
    xs = [dev(synth.gaussian_spinor(DIMS, k, nrhs=2)) for k in range(4)]
    refs = [torch.empty_like(x) for x in xs]
    for x, ref in zip(xs, refs):
        CALLS[name](ctx, x, ref)
    outs = [torch.zeros_like(x) for x in xs]
    s1 = torch.cuda.Stream()
    s2 = torch.cuda.Stream() if second == "other" else torch.cuda.default_stream()
    for s in (s1, s2):  # each stream's graph exists
        with torch.cuda.stream(s):
            CALLS[name](ctx, xs[0], outs[0])
    outs[0].zero_()
    torch.cuda.synchronize()
    for k, s in enumerate((s1, s2, s1, s2)):
        with torch.cuda.stream(s):
            if s is s1:
                busy(1)
            CALLS[name](ctx, xs[k], outs[k])
    for ref, out in zip(refs, outs):
        assert (host(out) == host(ref)).all()


def test_set_gauge_waits_for_calls_on_other_streams(busy):
    ctx = make()
    x = dev(synth.gaussian_spinor(DIMS, 1, nrhs=2))
    u2 = dev(synth.gauge_field(DIMS, 9, 0.5))
    f = [ctx.field(2, "f64") for _ in range(2)]
    f[0].load(x)
    outs = [torch.zeros_like(x) for _ in range(2)]
    refs = [torch.zeros_like(x) for _ in range(2)]
    s1 = torch.cuda.Stream()

    def go(res):
        with torch.cuda.stream(s1):
            ctx.apply_Hw(x, res[0], -RHO, prec="f64")
            ctx.dslash_field(f[0], f[1], -RHO)

    go(refs)
    f[1].store(refs[1], stream=s1)
    torch.cuda.synchronize()
    with torch.cuda.stream(s1):
        busy()
    go(outs)
    ctx.set_gauge(u2, stream=torch.cuda.Stream())
    f[1].store(outs[1], stream=s1)
    for ref, out in zip(refs, outs):
        assert (host(out) == host(ref)).all()
    for a in f:
        a.close()


@pytest.mark.parametrize("name", ["Hw", "net"])
def test_input_tensor_dropped_after_the_call(name, busy):
    """A call on a side stream returns before its work has begun; its input's memory is not handed out again to
    the current stream until that work is done."""
    ctx = make()
    psi = synth.gaussian_spinor(DIMS, 1, nrhs=2)
    ref, out = torch.empty_like(dev(psi)), torch.empty_like(dev(psi))
    s1 = torch.cuda.Stream()
    run = {"Hw": lambda x, o: ctx.apply_Hw(x, o, -RHO, prec="f32", stream=s1),
           "net": lambda x, o: ctx.net_apply(x, o, stream=s1)}[name]
    run(dev(psi), ref)
    torch.cuda.synchronize()
    x = dev(psi)
    torch.cuda.synchronize()
    with torch.cuda.stream(s1):
        busy()
    run(x, out)
    shape, kind = x.shape, x.dtype
    del x
    refill = [torch.zeros(shape, dtype=kind, device="cuda") for _ in range(8)]
    assert (host(out) == host(ref)).all()
    del refill
