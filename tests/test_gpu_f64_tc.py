"""FP64 mu-mode products on the tensor cores (contract_f64.cu) at the edges of their tiles: lines of
one chunk of 32 less, equal and more, lines past one accumulation segment of 256, position and
fibre counts around 64 and 128, odd rows; and the values that take its plain-FMA path.

Bounds, fixed beforehand: against the oracle 1e-12, as every FP64 action (each side's Padé factors are
within 6e-14 of the exact ones). A scaling by a power of two changes no digit of a slice, so those results are
equal bit by bit; the FMA path rounds each of K products, K 2^-53 of the sum of their magnitudes."""
import numpy as np
import pytest

from oracle import adr_oracle as O
from parity import assert_parity
from test_gpu_parity import adr, check_guards, guarded, make_case, torch

pytestmark = pytest.mark.gpu

# every one above the work from which FP64 contexts use the tensor cores (1.5e6 FMAs a pass)
DIMS = [(65, 400), (257, 127), (520, 60), (300, 130), (64, 64, 64), (127, 33, 65), (31, 129, 96), (130, 65, 67)]


def context(dims, scheme="lawson4", **kw):
    a, b, r, u0 = make_case(dims, b=(4.0,) * len(dims))
    ctx = adr.Context(dims, 2e-3, scheme, "fp64", **kw)
    ctx.set_coeffs(a, b, r)
    return ctx, a, b, r, u0


@pytest.mark.parametrize("dims", DIMS)
@pytest.mark.parametrize("c", [0.5, 1.0])
def test_exponential_against_the_oracle(dims, c):
    ctx, a, b, r, u0 = context(dims)
    ops = O.GridOps(O.ADRProblem(dims, a, b, r), 2e-3)
    fv, v = guarded(u0.shape, torch.float64, u0)
    fy, y = guarded(u0.shape, torch.float64)
    ctx.apply_exp(c, v, y)
    torch.cuda.synchronize()
    check_guards(fv)
    check_guards(fy)
    assert_parity(y.cpu().numpy(), ops.expA(c, u0), 1e-12, what=f"exp {dims} {c}")


@pytest.mark.parametrize("dims", [(257, 127), (64, 64, 64), (127, 33, 65)])
@pytest.mark.parametrize("k", [0, 1, 2])
def test_phi_against_the_oracle(dims, k):
    ctx, a, b, r, u0 = context(dims, "etd2rk")
    ops = O.GridOps(O.ADRProblem(dims, a, b, r), 2e-3)
    v = torch.tensor(u0, device="cuda")
    y = torch.empty_like(v)
    ctx.apply_phi(k, v, y)
    torch.cuda.synchronize()
    assert_parity(y.cpu().numpy(), ops.phi(k, 1.0, u0) if k else ops.expA(1.0, u0), 1e-12, what=f"phi_{k} {dims}")


@pytest.mark.parametrize("dims", [(300, 130), (127, 33, 65)])
def test_scales_and_special_values(dims):
    ctx, a, b, r, u0 = context(dims)
    v = torch.tensor(u0, device="cuda")
    y, z = torch.empty_like(v), torch.empty_like(v)
    ctx.apply_exp(0.5, v, y)
    for e in (-300, 300):                                  # the tensor cores, other scales
        ctx.apply_exp(0.5, v * 2.0 ** e, z)
        assert torch.equal(z, y * 2.0 ** e), e
    for e in (-800, 900):                                  # outside their range: plain FMAs
        ctx.apply_exp(0.5, v * 2.0 ** e, z)
        err = float(((z * 2.0 ** -e) - y).abs().max() / y.abs().max())
        assert err <= len(dims) * max(dims) * 2.0 ** -53, (e, err)
    ctx.apply_exp(0.5, torch.zeros_like(v), z)
    assert torch.count_nonzero(z) == 0
    bad = v.clone()
    bad.view(-1)[7] = float("nan")                         # every output depends on every input
    ctx.apply_exp(0.5, bad, z)
    assert torch.isnan(z).all()
    bad.view(-1)[7] = float("inf")
    ctx.apply_exp(0.5, bad, z)
    assert not torch.isfinite(z).any()
    ctx.apply_exp(0.5, v, z)
    ctx.synchronize()
    assert torch.equal(z, y)
