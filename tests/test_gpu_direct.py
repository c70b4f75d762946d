"""The register-streaming verification kernel (AUTO, no u requested) at the sizes where it can go wrong: edges of its
8-node column tiles and 16-row blocks, both depth variants, launch boundaries inside one ragged batch, faults, and a
state base that is only 16-byte aligned (its loads are 32 bytes wide)."""
import numpy as np
import pytest
import torch

from paper_2607_16673_b200 import binding as speca
from paper_2607_16673_b200 import synth
from gpu_util import DevProblem, TOL_FP32, oracle_verify, rel_err

pytestmark = pytest.mark.gpu


def check(prob, max_nodes, chain=False):
    dp = DevProblem(prob, route=speca.ROUTE_AUTO, max_nodes=max_nodes)
    dp.verify_chain() if chain else dp.verify_tree()
    assert dp.status_value() == 0
    e = rel_err(dp.o.cpu().numpy(), oracle_verify(prob))
    assert e <= TOL_FP32, (prob.name, e)


def tree(n, depth, rng):
    return synth.chain_parent(n) if n <= min(depth, 3) else synth.random_tree_parent(n, depth, 3, rng)


@pytest.mark.parametrize("depth", [8, 16])
@pytest.mark.parametrize("d_k,d_v", [(64, 64), (64, 32), (64, 96), (128, 128), (128, 256), (128, 320), (256, 256), (256, 64)])
def test_node_counts_at_tile_edges(d_k, d_v, depth):
    rng = np.random.default_rng(d_k + d_v + depth)
    top = 64 if d_k == 64 else 32
    for sizes in ([1, 7, 8, 3], [9, 15, 16, 1], [17, 23, 24, 25, 31, 32], [33, 48, 63, 64, 5]):
        if max(sizes) <= top:
            prob = synth.make_problem(d_k + sizes[0], 2, 3, d_k, d_v, [tree(n, depth, rng) for n in sizes], max_depth=depth,
                                      state_std=0.3, name=f"{d_k}x{d_v} {sizes} depth {depth}")
            prob.scale = 0.5
            check(prob, max(sizes))


@pytest.mark.parametrize("n", [1, 2, 8, 9, 16])
def test_chain_entry_point(n):
    prob = synth.make_problem(700 + n, 2, 4, 128, 128, [synth.chain_parent(n), synth.chain_parent(1)], max_depth=16)
    check(prob, 16, chain=True)


@pytest.mark.parametrize("L,B,d_k,d_v", [(3, 12, 128, 128), (3, 12, 128, 32), (3, 12, 256, 256), (2, 6, 256, 256)])
def test_batches_around_one_wave(L, B, d_k, d_v):
    """Between two and three units per SM (smaller CTAs), and unit counts whose value rows are split or not."""
    rng = np.random.default_rng(705 + d_v)
    top = 32 if d_k == 128 else 8
    parents = [tree(int(n), 6, rng) for n in np.linspace(1, top, B).round()]
    check(synth.make_problem(706 + d_v, L, 12, d_k, d_v, parents), top)


@pytest.mark.parametrize("d_k,B", [(64, 12), (128, 40)])
def test_ragged_batch_crosses_the_launch_boundaries(d_k, B):
    """Large enough for several launches by size; empty sequences, forests and every size class in one batch."""
    rng = np.random.default_rng(710 + d_k)
    forest = np.array([-1, -1, 0, -1, 1, 1, 2, 3, 3, 6], np.int32)
    parents = [np.zeros(0, np.int32), forest] + [tree(int(n), 8, rng) for n in np.linspace(1, 64, B - 2).round()]
    prob = synth.make_problem(711 + d_k, 10, 8, d_k, 64 if d_k == 64 else 128, parents)
    check(prob, 64)


def test_faults_skip_the_sequence():
    rng = np.random.default_rng(720)
    parents = [tree(12, 5, rng) for _ in range(4)]
    for kind, bit in (("parent", speca.STATUS_BAD_PARENT), ("depth", speca.STATUS_BAD_DEPTH), ("deep", speca.STATUS_TOO_DEEP),
                      ("many", speca.STATUS_TOO_MANY)):
        ps = list(parents)
        if kind == "deep":
            ps[1] = synth.chain_parent(12)
        if kind == "many":
            ps[1] = tree(20, 5, rng)
        prob = synth.make_problem(721, 2, 2, 128, 128, ps)
        good = oracle_verify(prob)
        s, e = int(prob.node_offsets[1]), int(prob.node_offsets[2])
        dp = DevProblem(prob, route=speca.ROUTE_AUTO, max_nodes=16)
        if kind == "parent":
            dp.parent[s + 3] = 7
        if kind == "depth":
            dp.depth[s + 3] += 1
        dp.verify_tree(with_depth=kind != "parent")
        assert dp.status_value() == bit, kind
        o = dp.o.cpu().numpy()
        keep = np.r_[0:s, e:prob.T]
        assert np.all(np.isnan(o[:, s:e])) and rel_err(o[:, keep], good[:, keep]) <= TOL_FP32


def test_state_base_of_sixteen_byte_alignment():
    prob = synth.make_problem(730, 2, 2, 128, 128, [synth.chain_parent(8), synth.chain_parent(5)])
    dp = DevProblem(prob, route=speca.ROUTE_AUTO, max_nodes=8)
    room = torch.zeros(dp.S.numel() + 64, device="cuda")
    view = room[4:4 + dp.S.numel()].view_as(dp.S)
    assert view.data_ptr() % 32 == 16
    view.copy_(dp.S)
    dp.S = view
    dp.verify_tree()
    assert dp.status_value() == 0 and rel_err(dp.o.cpu().numpy(), oracle_verify(prob)) <= TOL_FP32


@pytest.mark.parametrize("L,B,H,d_k,d_v,n,chain,serial", [
    (1, 4, 4, 64, 64, 3, True, True),            # a few short chains: the serial walk's work is less than the set-up here
    (1, 4, 4, 64, 64, 6, True, False),
    (6, 16, 16, 64, 64, 2, True, True),
    (6, 16, 16, 64, 64, 8, True, False),
    (6, 16, 16, 64, 32, 3, False, True),         # trees: only units this small, and the plan must not be the whole time
    (6, 16, 16, 64, 32, 5, False, False),
    (1, 2, 4, 64, 32, 1, False, False),
    (4, 64, 16, 256, 64, 1, False, True)])
def test_short_drafts_stay_with_the_serial_walk(L, B, H, d_k, d_v, n, chain, serial):
    parents = [synth.chain_parent(n)] * B
    prob = synth.make_problem(740 + n, L, H, d_k, d_v, parents, max_depth=8)
    out = {}
    for route in (speca.ROUTE_AUTO, speca.ROUTE_SERIAL):
        dp = DevProblem(prob, route=route, max_nodes=n)
        dp.verify_chain() if chain else dp.verify_tree()
        assert dp.status_value() == 0
        out[route] = dp.o
    assert torch.equal(out[speca.ROUTE_AUTO], out[speca.ROUTE_SERIAL]) == serial        # bit for bit: the same kernel
    assert float((out[speca.ROUTE_AUTO] - out[speca.ROUTE_SERIAL]).abs().max()) < 1e-5
    if L * B * H <= 64:
        assert rel_err(out[speca.ROUTE_AUTO].cpu().numpy(), oracle_verify(prob)) <= TOL_FP32


def test_one_large_tree_among_few_takes_the_others_along():
    """More nodes than a launch of this kernel could take: every sequence is walked serially, none twice or never."""
    rng = np.random.default_rng(750)
    prob = synth.make_problem(751, 1, 2, 64, 64, [tree(n, 8, rng) for n in (150, 9, 64)], max_depth=8)
    check(prob, 160)
    check(synth.make_problem(752, 1, 2, 64, 64, [tree(n, 8, rng) for n in (66, 9, 64)], max_depth=8), 160)


@pytest.mark.parametrize("route", [speca.ROUTE_SERIAL, speca.ROUTE_AUTO])
@pytest.mark.parametrize("n,bad", [(2, 0), (2, 3), (8, 0), (8, 3)])
def test_offsets_that_miss_the_ends_are_a_fault_on_every_route(n, bad, route):
    """Offsets that do not start at 0 or do not end at the number of nodes: the first or last chain is skipped, whichever
    kernel verifies the call (two nodes: the serial walk, eight: this one)."""
    prob = synth.make_problem(760 + n, 1, 4, 64, 64, [synth.chain_parent(n)] * 3)
    good = oracle_verify(prob)
    dp = DevProblem(prob, route=route, max_nodes=n)
    dp.node_offsets[bad] += 1 if bad == 0 else -1
    dp.verify_chain()
    assert dp.status_value() == speca.STATUS_BAD_OFFSETS
    skipped = slice(0, n) if bad == 0 else slice(2 * n, 3 * n)
    o = dp.o.cpu().numpy()
    assert np.isnan(o[:, skipped]).all()
    assert rel_err(np.delete(o, np.r_[skipped], 1), np.delete(good, np.r_[skipped], 1)) <= TOL_FP32
