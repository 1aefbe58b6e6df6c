"""Mixed-precision mu-mode products (contract_tc.cu) at the edges of their tiles: 64 lines a tile and 32 where 64
would leave SMs idle, ragged last tiles, extents off the 4 and 8 of the wide accesses, K of one chunk of 32, one
more, and the largest.

Bounds, fixed beforehand: 1e-6 against the oracle, as every mixed exponential."""
import pytest
from oracle import adr_oracle as O
from parity import assert_parity
from test_gpu_mixed import check_guards, ctx_for, guarded, make, np, torch

pytestmark = pytest.mark.gpu

# (32, 3) and (33, 512): 32 lines; (256, 160): both on one grid; the last three: 64 lines
DIMS = [(32, 3), (33, 512), (256, 160), (161, 63, 159), (33, 100, 300), (512, 20, 72)]


@pytest.mark.parametrize("dims", DIMS)
@pytest.mark.parametrize("c", [0.5, 1.0])
def test_exponential_against_the_oracle(dims, c):
    a, b, r = make(dims, b=(4.0,) * len(dims))
    v0 = 0.2 + 0.1 * np.random.default_rng(5).standard_normal(tuple(dims[::-1]))
    ctx = ctx_for(dims, 1e-3, "lawson4", a, b, r)
    ops = O.GridOps(O.ADRProblem(dims, a, b, r), 1e-3)
    fv, v = guarded(v0.shape, v0)
    fy, y = guarded(v0.shape)
    ctx.apply_exp(c, v, y)
    ctx.synchronize()
    check_guards(fv)
    check_guards(fy)
    assert_parity(y.cpu().numpy(), ops.expA(c, v.double().cpu().numpy()), 1e-6, what=f"exp {dims} {c}")
