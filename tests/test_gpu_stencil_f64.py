"""FP64 stencil (stencil_f64.cu) at the edges of its blocks and over what it leaves out: an odd x1 extent (one node a
thread) and an even one (two), rows shorter and longer than a block's 64 nodes, plane counts that end a
march early, Neumann faces, no advection term (b = 0), beta equal to b, and either output alone.

Bound, fixed beforehand: 1e-13 against the oracle, as every FP64 stencil test."""
import pytest

from oracle import adr_oracle as O
from parity import assert_parity
from test_gpu_parity import adr, check_guards, guarded, make_case, torch

pytestmark = pytest.mark.gpu

DIMS = [(5, 3), (63, 9), (64, 8), (66, 17), (129, 2), (5, 4, 3), (31, 9, 2), (62, 8, 33), (130, 7, 18)]


@pytest.mark.parametrize("dims", DIMS)
@pytest.mark.parametrize("b", [(0.0, 0.0, 0.0), (5.0, 0.0, -3.0)])
@pytest.mark.parametrize("form", ["flux", "adelta", "neumann"])
def test_F_and_g(dims, b, form):
    a, bb, r, u0 = make_case(dims, b=b[: len(dims)])
    kw = {"flux": {}, "adelta": dict(form="adelta"), "neumann": dict(bc="mixed", form="adelta")}[form]
    ctx = adr.Context(dims, 1e-3, "lawson4", "fp64", **kw)
    ctx.set_coeffs(a, bb, r)
    prob = O.ADRProblem(dims, a, bb, r, **kw)
    _, u = guarded(u0.shape, torch.float64, u0)
    for want in ("Fg", "F", "g"):
        fF, F = guarded(u0.shape, torch.float64)
        fg, g = guarded(u0.shape, torch.float64)
        ctx.eval_rhs(u, F if "F" in want else None, g if "g" in want else None)
        torch.cuda.synchronize()
        check_guards(fF)
        check_guards(fg)
        if "F" in want:
            assert_parity(F.cpu().numpy(), prob.F(u0), 1e-13, what=f"F {dims} {form}")
        if "g" in want:
            assert_parity(g.cpu().numpy(), prob.g(u0), 1e-13, what=f"g {dims} {form}")
