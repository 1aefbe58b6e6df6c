"""Fourier passes (periodic.cu) at the ends of the line lengths: rows as n/2 complex points down to n1 = 2, FP64 lines so
long that a block holds one of its two arrays at a time, columns of 2, and a third direction of 2, in FP64 and FP32.

Bounds, fixed beforehand: those of the shorter lines for the actions, 1e-12 (FP64), and 1e-5 (FP32: rounding of
each butterfly level, 12 at most a direction, 6e-8 each)."""
import pytest
from oracle import adr_oracle as O
from parity import assert_parity
from test_gpu_periodic import W, context, dev, host, np, torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,tol", [("fp64", 1e-12), ("fp32", 1e-5)])
@pytest.mark.parametrize("dims", [(2, 2), (4096, 4), (4, 1024), (2048, 2), (2, 4, 2), (64, 2, 16)])
def test_actions_match_oracle(dims, prec, tol):
    w, L, a, b = W.periodic_instance(dims, T=0.05, m=4)
    ctx = context(w, L, a, b, prec, scheme="etd2rk")
    ops = O.PeriodicOps(O.PeriodicProblem(dims, L, a, b, w.r_poly), w.tau)
    v = np.random.default_rng(3).standard_normal(w.u0.shape)
    x = dev(v, prec)
    for k in (0, 1, 2):
        y = torch.empty_like(x)
        ctx.apply_phi(k, x, y)
        ctx.synchronize()
        assert_parity(host(y), ops.phi(k, 1.0, host(x)) if k else ops.expA(1.0, host(x)), tol, what=f"{dims} {prec} {k}")
