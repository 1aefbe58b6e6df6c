"""FP64 exponentials (contract_f64.cu) whose factors and results leave the middle of the FP64 range: e^{tau A_mu} of 2^-480 and
2^-700 a direction, states scaled up and down, results that are subnormal or underflow, and sums that cancel.

Bounds, fixed beforehand. A scaling by a power of two changes no digit, so results in the normal range are equal bit by bit
and subnormal ones differ from the scaled result by their own rounding, 2^-1074. Lines below 2^-958 are summed by FMAs: N
roundings a direction, of 2^-53 of the sum or of 2^-1075. Against the oracle: each side's factors are
off by a few units of 2^-53 of tau ||A_mu|| (the exponent is that large), 16 of them are allowed. For a state that is odd
about the middle of x1 the exact sums vanish, and what is left is that error of the factors."""
import numpy as np
import pytest

from oracle import adr_oracle as O
from parity import assert_parity
from test_gpu_parity import adr, torch

pytestmark = pytest.mark.gpu

N, A = 128, 1.5


def setup(bits):
    tau = bits * np.log(2.0) / (A * np.pi ** 2)            # e^{tau A_mu} is about 2^-bits
    a = np.full((N + 2, N + 2), A)
    ctx = adr.Context((N, N), tau, "lawson4", "fp64")
    ctx.set_coeffs(a, (0.0, 0.0, 0.0), (0.0, 0.0, 0.0, 0.0))
    mf = O.MatrixFunctions(O.ADRProblem((N, N), a, (0.0, 0.0, 0.0), (0.0, 0.0, 0.0, 0.0)), tau)
    return ctx, mf, 16 * tau * 4 * A * (N + 1) ** 2 * 2.0 ** -53


def exp(ctx, u):
    v = torch.tensor(u, device="cuda")
    y = torch.empty_like(v)
    ctx.apply_exp(1.0, v, y)
    ctx.synchronize()
    return y.cpu().numpy()


# bits of decay a direction, scale of the reference state, scales of the others
@pytest.mark.parametrize("bits,ref,others", [(480, 0, (-450, -90, -30, 200, 400)), (700, 480, (450, 400, 350, -300)),
                                             (40, 0, (-900, -960, -990, -1000, 480))])
def test_scaled_states(bits, ref, others):
    ctx, mf, tol = setup(bits)
    u = np.random.default_rng(1).uniform(0.5, 1.0, (N, N))
    y0 = exp(ctx, np.ldexp(u, ref))
    want = mf.exp_action(1.0, np.ldexp(u, ref))
    assert np.isfinite(y0).all() and (y0 > 0).all()
    assert np.abs(y0 / want - 1.0).max() <= 2 * tol        # two directions
    for e in others:
        y = exp(ctx, np.ldexp(u, e))
        scaled = np.ldexp(y0, e - ref)
        if bits + 8 <= 958 + e:                            # both directions' lines are cut
            normal = scaled >= 2.0 ** -1022
            assert np.array_equal(y[normal], scaled[normal]), (bits, e)
            assert np.abs(y[~normal] - scaled[~normal]).max(initial=0.0) <= 2.0 ** -1074, (bits, e)
        else:                                              # below: N FMAs a result, each rounded
            assert (np.abs(y - scaled) <= 2 * N * 2.0 ** -53 * scaled + N * 2.0 ** -1074).all(), (bits, e)


@pytest.mark.parametrize("e", [0, -40, -300, -440, -490, -520])
def test_sums_that_cancel(e):
    ctx, mf, tol = setup(480)
    h = np.random.default_rng(3).uniform(0.5, 1.0, (N, N // 2))
    y = exp(ctx, np.ldexp(np.concatenate([h, -h[:, ::-1]], axis=1), e))
    emax = float(np.log2(max(np.abs(E).max() for E in mf.E_factors(1.0))))
    bound = 2 * (np.log2(N) + emax) + np.log2(tol) + e
    assert np.isfinite(y).all()
    worst = float(np.abs(y).max())
    assert worst == 0.0 or np.log2(worst) <= max(bound, -1073.0), (worst, bound)


def test_a_factor_out_of_range_concerns_no_other():
    """V_1 of a cell Peclet number of 0.92 on 400 nodes has entries of 2^460; a Lawson scheme applies e^{tau A_mu} only, whose
    entries are at most about 1: its passes stay on the tensor cores (kind 4 of a profiled step; 3: plain FMAs)."""
    dims, tau = (400, 60), 1e-6
    a, b, r = np.ones((62, 402)), (740.0, 0.0, 0.0), (0.0, 0.0, 1.0, -1.0)
    ctx = adr.Context(dims, tau, "lawson4", "fp64")
    ctx.set_coeffs(a, b, r)
    u = np.random.default_rng(5).standard_normal(dims[::-1])
    v = torch.tensor(u, device="cuda")
    y = torch.empty_like(v)
    ctx.apply_exp(0.5, v, y)
    kinds = [k for k, _ in ctx.profile_step(v)]
    ctx.synchronize()
    ops = O.GridOps(O.ADRProblem(dims, a, b, r), tau)
    assert_parity(y.cpu().numpy(), ops.expA(0.5, u), 1e-12, what="exp")
    assert 3 not in kinds and kinds.count(4) == 8, kinds
