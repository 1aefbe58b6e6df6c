"""Contexts on a device with little memory left: face weights, phi tables and cut factors are there for speed, and adr_set_coeffs
does without any of them that does not fit. The rest of the device is filled with one allocation that nothing touches; what
is left over shrinks from what the context would like to what it cannot do without (the nodal array and the dense factors).

Bounds, fixed beforehand: weights and phi factors formed in the kernels have the bits of the stored ones; the FMA kernel in
place of the cut factors rounds K times a sum, K 2^-53 of its terms a pass at most and 1e-13 in all for these grids."""
import pytest

from test_gpu_parity import W, adr, torch

pytestmark = pytest.mark.gpu

MB = 1 << 20


def fill(leave):
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    free = torch.cuda.mem_get_info()[0]
    return torch.empty(max(free - leave, 0), dtype=torch.uint8, device="cuda")


def problem(dims, prec):
    a = W.sine_product_coefficient(dims, c=0.4)
    dt = torch.float64 if prec == "fp64" else torch.float32
    u0 = torch.as_tensor(W.smooth_initial_state(dims, noise=1e-3, seed=11)).to(dt).cuda()
    b = (6.0, -4.0, 3.0)[: len(dims)] + (0.0,) * (3 - len(dims))
    return a, b, u0


def outputs(ctx, u0, scheme, tau):
    u, F, g, y = u0.clone(), torch.empty_like(u0), torch.empty_like(u0), torch.empty_like(u0)
    torch.cuda.synchronize()
    ctx.integrate(u, 0.0, 3 * tau, 3)
    ctx.eval_rhs(u0, F, g)
    if scheme == "etd2rk":
        ctx.apply_phi(2, u0, y)
    else:
        ctx.apply_exp(1.0, u0, y)
    ctx.synchronize()
    return [t.clone() for t in (u, F, g, y)]


@pytest.mark.parametrize("dims,scheme,prec,least", [
    ((128, 128, 128), "etd2rk", "fp64", 30), ((127, 96, 130), "lawson4", "fp64", 26), ((512, 96), "etd2rk", "fp64", 20),
    ((128, 128, 128), "etd2rk", "fp32", 20), ((128, 128, 128), "etd2rk", "bf16x3", 24)])
def test_new_coefficients(dims, scheme, prec, least):
    tau = 1e-3
    a, b, u0 = problem(dims, prec)
    r = (0.0, 0.0, 1.0, -1.0)

    def run(leave):
        ctx = adr.Context(dims, tau, scheme, prec)
        full = fill(leave) if leave else None
        before = torch.cuda.mem_get_info()[0]
        ctx.set_coeffs(a, b, r)
        used = before - torch.cuda.mem_get_info()[0]
        del full
        torch.cuda.empty_cache()
        out = outputs(ctx, u0, scheme, tau)
        ctx.close()
        return out, used

    run(0)                                                 # kernels loaded
    want, used = run(0)
    lefts = sorted({least * MB, *(int(least * MB + (used - least * MB) * f) for f in (0.25, 0.5, 0.75, 1.0))}, reverse=True)
    spent = []
    for leave in lefts:
        got, now = run(leave)
        spent.append(now)
        for x, y in zip(got, want):
            if prec == "fp64" and now < used:
                assert float((x - y).norm() / y.norm()) <= 1e-13, leave
            else:
                assert torch.equal(x, y), leave
    assert min(spent) < used, (used, spent)                # something was done without
