"""Small grids, FP64 and FP32 (contract_small_kernel in contract_simt.cu, launches that start before their predecessor
ends): outputs off the 8 and 16 of a block, K off the quarters that four lanes take, the longest K of this kernel (512)
and one more, and steps in which every launch depends on the one before it.

Bounds, fixed beforehand, are those of the larger grids: exponentials 1e-12 and 1e-6 against the oracle, phi
actions and runs 1e-12 and 2e-5."""
import pytest

from oracle import adr_oracle as O
from parity import assert_parity
from test_gpu_parity import DTYPES, check_guards, context, guarded, make_case, torch

pytestmark = pytest.mark.gpu

DIMS = [(5, 7), (32, 33), (512, 8), (9, 513), (4, 6, 5), (40, 31, 3)]


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("dims", DIMS)
def test_actions_and_steps(dims, prec):
    a, b, r, u0 = make_case(dims, b=(4.0, -3.0, 2.0)[: len(dims)])
    tau, dt, m = 1e-3, DTYPES[prec], 11
    exp_tol, tol = (1e-12, 1e-12) if prec == "fp64" else (1e-6, 2e-5)
    ops = O.GridOps(O.ADRProblem(dims, a, b, r), tau)
    ctx = context(dims, tau, "etd2rk", prec, a, b, r)
    fv, v = guarded(u0.shape, dt, u0)
    fy, y = guarded(u0.shape, dt)
    vin = v.double().cpu().numpy()
    for k in (0, 1, 2):
        ctx.apply_phi(k, v, y)
        torch.cuda.synchronize()
        check_guards(fv)
        check_guards(fy)
        ref = ops.phi(k, 1.0, vin) if k else ops.expA(1.0, vin)
        assert_parity(y.cpu().numpy(), ref, tol if k else exp_tol, what=f"phi{k} {dims} {prec}")
    ctx.integrate(v, 0.0, m * tau, m)
    torch.cuda.synchronize()
    check_guards(fv)
    assert_parity(v.cpu().numpy(), O.integrate(ops, vin, m, "etd2rk"), tol, what=f"etd2rk {dims} {prec}")
