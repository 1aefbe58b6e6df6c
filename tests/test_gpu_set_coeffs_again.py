"""New coefficients for a context whose steps are still in flight: adr_set_coeffs rewrites buffers that those steps read,
and calls are ordered on the context's stream. Every run is compared with the same calls with a synchronisation between
them; both launch the same kernels on the same values, so the results are equal bit by bit.

The streams are non-blocking ones (torch.cuda.Stream), which nothing else orders against the library's uploads."""
import numpy as np
import pytest

from test_gpu_batch import W, adr, packed, torch

pytestmark = pytest.mark.gpu

# (dims, scheme, precision, extra arguments, steps of the first run: long enough to outlast the host's part of the second call)
GRIDS = [
    ((96, 96, 96), "etd2rk", "fp64", {}, 150),
    ((300, 200), "lawson4", "fp64", {}, 600),
    ((64, 64, 64), "lawson2a", "fp64", dict(bc="mixed", form="adelta"), 300),
    ((96, 96, 96), "lawson2b", "fp32", {}, 150),
    ((128, 96, 64), "etd2rk", "bf16x3", {}, 300),
    ((40, 36, 33), "etd2rk", "fp64", dict(phi_route="doubling"), 60),
]


def two_runs(make, first, second, u0, tau, m, wait):
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        u = torch.as_tensor(u0, device="cuda").clone()
    ctx = make(stream)
    first(ctx)
    stream.synchronize()
    ctx.integrate(u, 0.0, m * tau, m)
    if wait:
        stream.synchronize()
    second(ctx)
    ctx.integrate(u, 0.0, 5 * tau, 5)
    ctx.synchronize()
    out = u.clone()
    ctx.close()
    return out


def compare(*args):
    a, b = two_runs(*args, True), two_runs(*args, False)
    assert torch.isfinite(a).all()
    assert torch.equal(a, b)


@pytest.mark.parametrize("dims,scheme,prec,kw,m", GRIDS)
def test_single_grids(dims, scheme, prec, kw, m):
    tau, d = 1e-4, len(dims)
    dt = torch.float64 if prec == "fp64" else torch.float32

    def coeffs(c, b, r):
        a = W.sine_product_coefficient(dims, c=c)
        return lambda ctx: ctx.set_coeffs(a, (b,) * d, r)

    u0 = torch.as_tensor(W.smooth_initial_state(dims, noise=1e-3, seed=3)).to(dt)
    compare(lambda s: adr.Context(dims, tau, scheme, prec, stream=s, **kw),
            coeffs(0.5, 4.0, (0.0, 0.0, 1.0, -1.0)), coeffs(0.2, -3.0, (0.1, 0.0, 0.5, -1.0)), u0, tau, m)


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_periodic(prec):
    w, L, a, b = W.periodic_instance((256, 128), T=0.01, m=100)
    dt = torch.float64 if prec == "fp64" else torch.float32

    def coeffs(f):
        return lambda ctx: ctx.set_coeffs_periodic([f * x for x in a], [-f * x for x in b], w.r_poly)

    compare(lambda s: adr.Context(w.dims, w.tau, "lawson2a", prec, stream=s, periodic=True, length=L),
            coeffs(1.0), coeffs(0.5), torch.as_tensor(np.ascontiguousarray(w.u0)).to(dt), w.tau, 400)


@pytest.mark.parametrize("prec", ["fp64", "fp32", "bf16x3"])
def test_batches(prec):
    ws = W.batch_instances([(100, 96), (64, 129), (200, 180)], T=0.01, scheme="lawson4")
    _, u0 = packed(ws, "fp64" if prec == "fp64" else "fp32")

    def coeffs(f):
        def put(ctx):
            for i, w in enumerate(ws):
                ctx.set_coeffs(f * w.a_nodes, w.b, w.r_poly, instance=i)
        return put

    compare(lambda s: adr.Context(None, ws[0].tau, "lawson4", prec, stream=s, batch_dims=[w.dims for w in ws], batch_tile=64),
            coeffs(1.0), coeffs(0.6), u0.clone(), ws[0].tau, 400)
