"""The substitution kernel with split operands serves the fp32-grade calls that ask for u (without u the same routes run
another kernel): parity, the chain entry point, faults in device memory and an expired wait, with u requested."""
import ctypes

import numpy as np
import pytest

from paper_2607_16673_b200 import binding as speca
from paper_2607_16673_b200 import synth
from gpu_util import DevProblem, TOL_FP32, oracle_verify, rel_err

pytestmark = pytest.mark.gpu

ROUTES = [speca.ROUTE_FACTORIZED, speca.ROUTE_AUTO]


def cpu(t):
    return t.detach().cpu().numpy()


def check(prob, route, max_nodes, chain=False):
    dp = DevProblem(prob, route=route, want_u=True, max_nodes=max_nodes)
    (dp.verify_chain if chain else dp.verify_tree)()
    assert dp.status_value() == 0
    assert rel_err(cpu(dp.o), oracle_verify(prob)) <= TOL_FP32
    ds = DevProblem(prob, route=speca.ROUTE_SERIAL, want_u=True, max_nodes=max_nodes)
    (ds.verify_chain if chain else ds.verify_tree)()
    assert rel_err(cpu(dp.u), cpu(ds.u)) <= TOL_FP32


@pytest.mark.parametrize("route", ROUTES)
@pytest.mark.parametrize("d_k,d_v,depth", [(128, 128, 8), (128, 256, 8), (256, 256, 8), (128, 256, 16), (256, 128, 16)])
def test_outputs_and_corrected_values(d_k, d_v, depth, route):
    rng = np.random.default_rng(d_k + d_v + depth)
    top = 64 if d_k == 128 and depth == 8 else 32
    sizes = [top, 1, 17, 16, 0, top - 1, 33 if top == 64 else 9, 8]
    parents = [synth.random_tree_parent(n, depth, 4, rng) if n > 3 else synth.chain_parent(n) for n in sizes]
    prob = synth.make_problem(1500 + d_k + depth, 3, 4, d_k, d_v, parents, max_depth=depth, state_std=0.3)
    prob.scale = 0.5
    check(prob, route, top)


@pytest.mark.parametrize("route", ROUTES)
def test_chain_entry_point(route):
    chains = [synth.chain_parent(n) for n in (8, 1, 5, 7, 8)]
    check(synth.make_problem(1520, 2, 3, 128, 256, chains), route, 16, chain=True)


@pytest.mark.parametrize("route", ROUTES)
def test_faults_skip_the_sequence(route):
    rng = np.random.default_rng(1530)
    prob = synth.make_problem(1531, 2, 2, 128, 128, [synth.random_tree_parent(12, 5, 3, rng) for _ in range(4)])
    good = oracle_verify(prob)
    s1, e1 = int(prob.node_offsets[1]), int(prob.node_offsets[2])
    prob.parent[s1 + 3] = 7
    dp = DevProblem(prob, route=route, want_u=True, max_nodes=16)
    dp.verify_tree(with_depth=False)
    assert dp.status_value() == speca.STATUS_BAD_PARENT
    o, u = cpu(dp.o), cpu(dp.u)
    assert np.all(np.isnan(o[:, s1:e1])) and np.all(np.isnan(u[:, s1:e1]))
    keep = np.r_[0:s1, e1:prob.T]
    assert rel_err(o[:, keep], good[:, keep]) <= TOL_FP32 and np.isfinite(u[:, keep]).all()


def test_expired_wait_is_reported_and_the_context_stays_usable():
    """One CTA's first state slice is never requested (the library's test hook): its bounded waits run out, the kernel
    returns, the status word carries TIMEOUT, and the next call works."""
    rng = np.random.default_rng(1540)
    prob = synth.make_problem(1541, 2, 4, 128, 128, synth.ragged_tree_batch(rng, 3, 4, 20, 8))
    dp = DevProblem(prob, route=speca.ROUTE_FACTORIZED, want_u=True, max_nodes=64)
    hook = speca.lib().speca_test_withhold_first_load
    hook.argtypes, hook.restype = [ctypes.c_int], None
    hook(1)
    try:
        dp.verify_tree()
        assert dp.status_value() & speca.STATUS_TIMEOUT
    finally:
        hook(0)
    dp.status.zero_()
    dp.o.fill_(float("nan"))
    dp.verify_tree()
    assert dp.status_value() == 0
    assert rel_err(cpu(dp.o), oracle_verify(prob)) <= TOL_FP32
