"""Calls of a few units, whose topology the verification kernel checks itself, on both sides of the number of sequences up to
which it does: outputs of the good sequences, and what is reported of the bad ones."""
import numpy as np
import pytest
import torch

from paper_2607_16673_b200 import binding as speca
from paper_2607_16673_b200 import synth
from gpu_util import DevProblem, TOL_FP32, oracle_verify, rel_err

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("with_depth", [False, True])
@pytest.mark.parametrize("B,d_k,depth", [(1, 128, 8), (6, 256, 16), (19, 128, 8), (20, 128, 16), (20, 256, 8), (21, 128, 8)])
def test_good_and_bad_sequences(B, d_k, depth, with_depth):
    rng = np.random.default_rng(900 + B + d_k)
    top = 64 if d_k == 128 else 32
    parents = [synth.random_tree_parent(int(n), depth, 4, rng) for n in rng.integers(1, top + 1, B)]
    parents[-1] = synth.random_tree_parent(top, depth, 4, rng)
    if B > 4:
        parents[2] = np.zeros(0, np.int32)
    prob = synth.make_problem(901 + B, 1, 3, d_k, 128, parents, max_depth=depth)
    ref, offs = oracle_verify(prob), prob.node_offsets
    bad = {}                                           # sequence -> what is wrong with it
    if B > 4:
        bad[1] = speca.STATUS_BAD_PARENT
        if with_depth:
            bad[3] = speca.STATUS_BAD_DEPTH
    for broken in (False, True) if bad else (False,):
        dp = DevProblem(prob, route=speca.ROUTE_EFFECTIVE, max_nodes=top)
        if broken:
            dp.parent[offs[1] + len(parents[1]) - 1] = len(parents[1])
            if 3 in bad:
                dp.depth[offs[3]] += 1
        dp.verify_tree(with_depth)
        want, skip = (sum(bad.values()), bad) if broken else (0, {})
        assert dp.status_value() == want
        got = dp.o.cpu().numpy()
        for b in range(B):
            o = got[:, offs[b]:offs[b + 1]]
            if b in skip:
                assert np.isnan(o).all()
            elif o.size:
                assert rel_err(o, ref[:, offs[b]:offs[b + 1]]) <= TOL_FP32


def test_sequences_beyond_the_limits_of_the_call():
    """One node too many, one level too many: reported and left alone, the neighbours are not."""
    for parents, nodes, code in (([synth.chain_parent(5), synth.random_tree_parent(33, 8, 4, np.random.default_rng(1)), synth.chain_parent(7)],
                                  32, speca.STATUS_TOO_MANY),
                                 ([synth.chain_parent(8), synth.chain_parent(9), synth.chain_parent(1)], 32, speca.STATUS_TOO_DEEP)):
        prob = synth.make_problem(950, 1, 2, 128, 256, parents, max_depth=8)
        ref, offs = oracle_verify(prob), prob.node_offsets
        dp = DevProblem(prob, route=speca.ROUTE_EFFECTIVE, max_nodes=nodes)
        dp.verify_tree()
        assert dp.status_value() == code
        got = dp.o.cpu().numpy()
        assert np.isnan(got[:, offs[1]:offs[2]]).all()
        assert rel_err(got[:, :offs[1]], ref[:, :offs[1]]) <= TOL_FP32 and rel_err(got[:, offs[2]:], ref[:, offs[2]:]) <= TOL_FP32
