"""FP64 actions of states that are localised where the factors are badly scaled: V_mu = diag(rho^i) S, so the columns of
V_mu^-1 differ by kappa(V_mu), and a pulse at the end where they are small meets only the small ones. A sum of FP64
products does not mind (each keeps its 53 bits); one that holds the factor's rows and the state's lines in fixed point does.

Bounds, fixed beforehand: 1e-12 against the oracle, as every FP64 action (the oracle itself is within 7e-14 of 80-bit
sums on these problems)."""
import numpy as np
import pytest

from oracle import adr_oracle as O
from parity import assert_parity
from test_gpu_parity import adr, torch

pytestmark = pytest.mark.gpu


def pulse(dims, centre, width=0.05):
    out = np.ones(())
    for n in dims:                                         # x1 fastest
        x = np.arange(1, n + 1) / (n + 1.0)
        out = np.exp(-((x - centre) / width) ** 2).reshape((n,) + (1,) * out.ndim) * out
    return out


def problem(dims, b, tau, scheme):
    a = np.full([n + 2 for n in dims[::-1]], 1.5)
    b = tuple(float(v) for v in b) + (0.0,) * (3 - len(dims))
    r = (0.0, 0.0, 1.0, -1.0)
    ctx = adr.Context(dims, tau, scheme, "fp64")
    ctx.set_coeffs(a, b, r)
    return ctx, O.GridOps(O.ADRProblem(dims, a, b, r), tau)


@pytest.mark.parametrize("dims,b,centre", [((128, 128), (10, 10), 0.2), ((128, 128), (30, 0), 0.2), ((128, 128), (50, 0), 0.1),
                                           ((128, 128), (60, 0), 0.2), ((128, 128), (80, 0), 0.1), ((128, 128), (0, -60), 0.85),
                                           ((300, 40), (50, 20), 0.1), ((65, 40, 33), (0, 0, 30), 0.2),
                                           ((33, 65, 40), (10, 30, -10), 0.3)])
def test_pulses(dims, b, centre):
    ctx, ops = problem(dims, b, 2e-3, "etd2rk")
    u0 = pulse(dims, centre)
    v = torch.tensor(u0, device="cuda")
    y = torch.empty_like(v)
    for k in (0, 1, 2):
        ctx.apply_phi(k, v, y)
        ctx.synchronize()
        assert_parity(y.cpu().numpy(), ops.phi(k, 1.0, u0) if k else ops.expA(1.0, u0), 1e-12, what=f"phi_{k} {dims} {b}")


@pytest.mark.parametrize("dims,b,tau", [((128, 128), (60, -40), 1e-2), ((300, 70), (80, 10), 5e-3), ((40, 66, 65), (30, -60, 10), 1e-2)])
def test_exponentials_with_columns_of_several_sizes(dims, b, tau):
    """Advection that carries the state out of the box within a step or two: the columns of e^{c tau A_1} differ, too, and
    the stage combinations follow those passes."""
    ctx, ops = problem(dims, b, tau, "lawson2b")
    columns = np.abs(ops.mf.E_factors(1.0)[0]).max(axis=0)
    assert columns.max() > 16 * columns.min()
    u0 = pulse(dims, 0.5, 0.2) + 1e-3 * np.random.default_rng(2).standard_normal(dims[::-1])
    v = torch.tensor(u0, device="cuda")
    y = torch.empty_like(v)
    for c in (0.5, 1.0):
        ctx.apply_exp(c, v, y)
        ctx.synchronize()
        assert_parity(y.cpu().numpy(), ops.expA(c, u0), 1e-12, what=f"exp {dims} {c}")
    ctx.integrate(v, 0.0, 2 * tau, 2)
    ctx.synchronize()
    assert_parity(v.cpu().numpy(), O.integrate(ops, u0, 2, "lawson2b"), 1e-12, what=f"lawson2b {dims}")
