"""The effective-query kernel where its buffers change hands: units of up to 32 nodes (two buffers of M) next to
larger ones (one), several units per CTA, one and two value tiles, both key widths and depth variants, o and u walks, and
the rule without erase."""
import numpy as np
import pytest
import torch

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


def device_problem(seed, L, H, d_k, d_v, parents, depth):
    """A batch too large for the oracle as a whole: inputs made on the device, outputs of two routes, the same units of both
    for the oracle."""
    offs = np.concatenate([[0], np.cumsum([len(p) for p in parents])]).astype(np.int32)
    T, B = int(offs[-1]), len(parents)
    parent = np.concatenate(parents).astype(np.int32)
    S = synth.device_state(seed, L, B, H, d_k, d_v, 0.3, "cuda")
    q, k, v, al, be = synth.device_records(seed + 1, L, T, H, d_k, d_v, "cuda")
    dev = lambda a: torch.from_numpy(a).cuda()
    out = {}
    for route in (speca.ROUTE_EFFECTIVE, speca.ROUTE_SERIAL):
        dims = speca.Dims(L, B, H, d_k, d_v, 1.0, depth, max(len(p) for p in parents), route)
        o = torch.full((L, T, H, d_v), float("nan"), device="cuda")
        status = torch.zeros(1, dtype=torch.int32, device="cuda")
        speca.verify_tree(dims, S, q, k, v, al, be, dev(offs), T, dev(parent), None, o, None, speca.alloc_workspace(dims, T), status)
        assert int(status) == 0
        out[route] = o
    return S, (q, k, v, al, be), offs, parent, out


@pytest.mark.parametrize("d_k,d_v,depth,L,B,H", [
    (256, 256, 8, 24, 8, 8), (256, 128, 16, 24, 8, 8), (128, 256, 16, 24, 8, 8), (128, 128, 8, 24, 8, 8),
    # four heads of a sequence at a time from 128 units per SM on
    (128, 128, 16, 24, 50, 16), (256, 128, 8, 24, 50, 16)])
def test_the_form_for_large_calls(d_k, d_v, depth, L, B, H):
    """From eight units per SM on the kernel is launched plainly and walks its units otherwise: all units against the serial
    walk, a sample against the oracle."""
    rng = np.random.default_rng(d_k + d_v + depth)
    top = 64 if d_k == 128 else 32
    sizes = [top, 1, 17, 16, top // 2 + 1, 8, top, 31][:min(B, 8)]
    parents = [tree(n, depth, rng) for n in sizes * (B // 8) + sizes[:B % 8]]
    S, rec, offs, parent, out = device_problem(870 + d_k + depth, L, H, d_k, d_v, parents, depth)
    o, ref = out[speca.ROUTE_EFFECTIVE], out[speca.ROUTE_SERIAL]
    rms = float(ref.pow(2).mean().sqrt())
    assert float(((o - ref).abs() / (ref.abs() + rms)).max()) <= TOL_FP32
    host = [x.view(torch.int16) if x.dtype == torch.bfloat16 else x for x in rec]
    for l, b, h in zip(rng.integers(0, L, 6), rng.integers(0, B, 6), rng.integers(0, H, 6)):
        s, e = int(offs[b]), int(offs[b + 1])
        args = [np.ascontiguousarray(x[l:l + 1, s:e, h:h + 1].cpu().numpy()) for x in host]
        args = [a.view(np.uint16) if a.dtype == np.int16 else a for a in args]
        r = oracle.verify_tree(S[l:l + 1, b:b + 1, h:h + 1].cpu().numpy(), *args, np.array([0, e - s], np.int32), parent[s:e])
        assert rel_err(o[l, s:e, h].cpu().numpy(), r[0, :, 0]) <= TOL_FP32


@pytest.mark.parametrize("d_v", [128, 256])
def test_ring_slots_in_the_form_for_large_calls(d_v):
    rng = np.random.default_rng(880)
    sizes = [64, 1, 32, 33, 8, 16, 64, 17, 48, 49, 31, 15, 2]
    prob = synth.make_problem(881, 8, 4, 128, d_v, [tree(n, 8, rng) for n in sizes * 4], state_std=0.3)
    dp = DevProblem(prob, route=speca.ROUTE_EFFECTIVE, want_u=True, max_nodes=64)
    ds = DevProblem(prob, route=speca.ROUTE_SERIAL, want_u=True, max_nodes=64)
    dp.verify_tree()
    ds.verify_tree()
    assert dp.status_value() == 0 and rel_err(dp.o.cpu().numpy(), ds.o.cpu().numpy()) <= TOL_FP32
    o, u = dp.o.clone(), dp.u.clone()
    for _ in range(40):
        dp.o.zero_(); dp.u.zero_()
        dp.verify_tree()
        assert bool((dp.o == o).all()) and bool((dp.u == u).all())
