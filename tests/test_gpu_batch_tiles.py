"""Batched contractions at the edges of their tiles. Mixed (batch_tc.cu): 64 lines and 128 outputs a tile, K chunks of 32,
column groups of four, instances of one tile beside instances of many, more tiles than the ring of
tile descriptors holds. FP64 (batch2d.cu): the kernels for tiles up to 32, 64 and 128.

Bounds, fixed beforehand, are those of the other batched mixed tests: actions 1e-6 and runs 1e-5 against the oracle. The
tile shapes accumulate in one order, so those results are equal bit by bit."""
import pytest
from oracle import adr_oracle as O
from parity import assert_parity
from test_gpu_batch import W, batch_context, check_guards, np, packed, torch, unpack

pytestmark = pytest.mark.gpu

EDGES = [(2, 2), (3, 256), (256, 3), (63, 128), (64, 129), (65, 127), (128, 64), (129, 65), (255, 256), (31, 33), (36, 100)]


def test_mixed_action_and_steps():
    ws = W.batch_instances(EDGES * 2, scheme="lawson4")
    ctx = batch_context(ws, "bf16x3", "lawson4")
    rng = np.random.default_rng(2)
    _, v = packed(ws, "fp32", [rng.standard_normal(w.dims[::-1]) for w in ws])
    fy, y = packed(ws, "fp32", [np.zeros(w.dims[::-1]) for w in ws])
    ctx.apply_exp(0.5, v, y)
    fu, u = packed(ws, "fp32")
    ctx.integrate(u, 0.0, 4 * ws[0].tau, 4)
    ctx.synchronize()
    check_guards(fy)
    check_guards(fu)
    for w, vin, got, end in zip(ws, unpack(ws, v), unpack(ws, y), unpack(ws, u)):
        ops = O.GridOps(O.ADRProblem(w.dims, w.a_nodes, w.b, w.r_poly), w.tau)
        assert_parity(got, ops.expA(0.5, vin), 1e-6, what=("exp", w.name))
        assert_parity(end, O.integrate(ops, w.u0, 4, "lawson4"), 1e-5, what=("lawson4", w.name))


def test_fp64_tiles_give_equal_bits():
    ws = W.batch_instances([(5, 33), (32, 64), (65, 31), (100, 129)], scheme="etd2rk")
    outs = []
    for tile in (0, 32, 64, 128):
        ctx = batch_context(ws, "fp64", "etd2rk", tile=tile)
        full, u = packed(ws, "fp64")
        ctx.integrate(u, 0.0, 3 * ws[0].tau, 3)
        ctx.synchronize()
        check_guards(full)
        outs.append(u.clone())
    assert all(torch.equal(o, outs[0]) for o in outs)
