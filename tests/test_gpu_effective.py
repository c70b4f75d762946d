"""The effective-query kernel where its buffers change hands: units of up to 32 nodes (two buffers of x and of M) next to
larger ones (one), several units per CTA, one and two value tiles, both key widths and depth variants, o and u walks, and
the rule without erase."""
import numpy as np
import pytest

import oracle
from paper_2607_16673_b200 import binding as speca
from paper_2607_16673_b200 import synth
from gpu_util import DevProblem, TOL_FP32, oracle_verify, rel_err

pytestmark = pytest.mark.gpu


def tree(n, depth, rng):
    return synth.chain_parent(n) if n <= 3 else synth.random_tree_parent(n, depth, 4, rng)


@pytest.mark.parametrize("want_u", [False, True])
@pytest.mark.parametrize("depth", [8, 16])
@pytest.mark.parametrize("d_k,d_v", [(128, 128), (128, 256), (256, 128), (256, 256)])
def test_small_and_large_units_in_turn(d_k, d_v, depth, want_u):
    rng = np.random.default_rng(d_k + d_v + depth)
    top = 64 if d_k == 128 else 32
    sizes = [64, 1, 32, 33, 8, 16, 64, 0, 17, 48, 49, 31, 15, 2] if top == 64 else [32, 1, 16, 17, 8, 31, 0, 32, 9, 15, 2, 25]
    parents = [tree(n, depth, rng) if n else np.zeros(0, np.int32) for n in sizes * 4]
    # 56 (48) sequences x 3 heads x 4 layers: four to five units per CTA, one head at a time
    prob = synth.make_problem(800 + d_k + d_v, 4, 3, d_k, d_v, parents, max_depth=depth, state_std=0.3)
    prob.scale = 0.5
    dp = DevProblem(prob, route=speca.ROUTE_EFFECTIVE, want_u=want_u, max_nodes=top)
    dp.verify_tree()
    assert dp.status_value() == 0
    assert rel_err(dp.o.cpu().numpy(), oracle_verify(prob)) <= TOL_FP32
    if want_u:
        ds = DevProblem(prob, route=speca.ROUTE_SERIAL, want_u=True, max_nodes=top)
        ds.verify_tree()
        assert rel_err(dp.u.cpu().numpy(), ds.u.cpu().numpy()) <= TOL_FP32


@pytest.mark.parametrize("want_u", [False, True])
@pytest.mark.parametrize("d_k", [128, 256])
@pytest.mark.parametrize("L,B,H", [(1, 1, 1), (2, 7, 5), (3, 21, 3), (1, 37, 4), (4, 10, 5)])
def test_heads_split_by_value_tile(L, B, H, d_k, want_u):
    """Unit counts on both sides of every bound at which a head of two value tiles counts as two units."""
    rng = np.random.default_rng(840 + B)
    top = 64 if d_k == 128 else 32
    parents = [tree(int(n), 8, rng) for n in np.linspace(top, 1, B).round()]
    prob = synth.make_problem(841 + B, L, H, d_k, 256, parents, max_depth=8, state_std=0.3)
    dp = DevProblem(prob, route=speca.ROUTE_EFFECTIVE, want_u=want_u, max_nodes=top)
    dp.verify_tree()
    assert dp.status_value() == 0
    assert rel_err(dp.o.cpu().numpy(), oracle_verify(prob)) <= TOL_FP32
    if want_u:
        ds = DevProblem(prob, route=speca.ROUTE_SERIAL, want_u=True, max_nodes=top)
        ds.verify_tree()
        assert rel_err(dp.u.cpu().numpy(), ds.u.cpu().numpy()) <= TOL_FP32


def test_rule_without_erase():
    rng = np.random.default_rng(820)
    prob = synth.make_problem(821, 2, 4, 128, 256, [tree(n, 8, rng) for n in (40, 7, 64)])
    dp = DevProblem(prob, route=speca.ROUTE_EFFECTIVE, max_nodes=64, rule=speca.RULE_GATED_NO_ERASE)
    dp.verify_tree()
    assert dp.status_value() == 0
    oracle.set_rule(speca.RULE_GATED_NO_ERASE)
    try:
        ref = oracle_verify(prob)
    finally:
        oracle.set_rule(speca.RULE_GATED_DELTA)
    assert rel_err(dp.o.cpu().numpy(), ref) <= TOL_FP32


@pytest.mark.parametrize("d_v", [128, 256])
def test_ring_slots_are_read_before_they_are_refilled(d_v):
    """Many units per CTA from a state that L2 holds (the second walk of a unit with u requested reads it there): a ring slot
    comes round again as fast as it can.  Every repetition must give the first one's bits."""
    rng = np.random.default_rng(830)
    sizes = [64, 1, 32, 33, 8, 16, 64, 17, 48, 49, 31, 15, 2]
    prob = synth.make_problem(831, 4, 3, 128, d_v, [tree(n, 8, rng) for n in sizes * 4], state_std=0.3)
    dp = DevProblem(prob, route=speca.ROUTE_EFFECTIVE, want_u=True, max_nodes=64)
    dp.verify_tree()
    assert dp.status_value() == 0 and rel_err(dp.o.cpu().numpy(), oracle_verify(prob)) <= TOL_FP32
    o, u = dp.o.clone(), dp.u.clone()
    for _ in range(40):
        dp.o.zero_(); dp.u.zero_()
        dp.verify_tree()
        assert bool((dp.o == o).all()) and bool((dp.u == u).all())
