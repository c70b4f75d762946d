"""Small-tree verification with rows, steps, nodes and columns of very different magnitudes.  The products of larger trees work
on fp16 pairs scaled by row of the state and by node, 32 columns at a time: a power of two on a row of the state and its values,
or on a query, must come out as that power of two and nothing else, and a column that is much larger than the others of its 32
must not cost those their bits."""
import numpy as np
import pytest
import torch

from paper_2607_16673_b200 import synth
from gpu_util import DevProblem, TOL_FP32, oracle_verify, rel_err

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d_k,d_v,n,depth", [(64, 64, 8, 8), (64, 64, 17, 8), (64, 96, 32, 16), (64, 64, 33, 8), (64, 64, 64, 8),
                                             (128, 128, 24, 8), (128, 256, 32, 6), (256, 64, 25, 8)])
def test_powers_of_two_go_through(d_k, d_v, n, depth):
    rng = np.random.default_rng(n + d_k + d_v)
    prob = synth.make_problem(70 + n, 1, 3, d_k, d_v, [synth.random_tree_parent(n, depth, 4, rng), synth.random_tree_parent(max(1, n - 7), depth, 4, rng)],
                              max_depth=depth, state_std=0.3)
    # a step of 32 columns that is much larger than the others, and one that is zero
    prob.S0[..., :32] *= 2.0 ** 12
    prob.S0[:, :, 1, :, 32:64] = 0.0
    dp = DevProblem(prob, max_nodes=n)
    base = dp.verify_tree().clone()
    assert dp.status_value() == 0
    assert rel_err(base.cpu().numpy(), oracle_verify(prob)) <= TOL_FP32
    rows = torch.from_numpy(2.0 ** rng.integers(-50, 51, d_v)).float().cuda()
    nodes = torch.from_numpy(2.0 ** rng.integers(-20, 21, dp.T)).float().cuda()
    dp.S *= rows[:, None]
    dp.v = (dp.v.float() * rows).to(torch.bfloat16)
    dp.q = (dp.q.float() * nodes[None, :, None, None]).to(torch.bfloat16)
    dp.verify_tree()
    assert dp.status_value() == 0
    assert torch.equal(dp.o, base * rows * nodes[None, :, None, None])


SHAPES = [(64, 64, 16, 8), (64, 64, 17, 8), (64, 96, 32, 16), (64, 64, 40, 8), (64, 64, 64, 16), (128, 128, 24, 8), (128, 256, 32, 6),
          (256, 64, 25, 8)]
# Every product loses at most 2^-22 of itself (two operands of 23 bits), and sums of up to 64 n random ones in fp32 no more
TOL_PRODUCTS = 2.0 ** -22


def state_only(d_k, d_v, n, depth):
    """A problem whose outputs come from the state alone."""
    rng = np.random.default_rng(n + d_k + d_v)
    trees = [synth.random_tree_parent(max(1, m), depth, 4, rng) for m in (n, n - 7, n)]
    prob = synth.make_problem(90 + n, 1, 3, d_k, d_v, trees, max_depth=depth, state_std=0.5)
    prob.v[:] = 0
    return prob


def error_norm(prob, n):
    dp = DevProblem(prob, max_nodes=n)
    dp.verify_tree()
    assert dp.status_value() == 0
    ref = oracle_verify(prob)
    return float(np.linalg.norm(dp.o.cpu().numpy().astype(np.float64) - ref) / np.linalg.norm(ref))


@pytest.mark.parametrize("d_k,d_v,n,depth", SHAPES)
@pytest.mark.parametrize("exponent", [12, 20, 26, 27, 28, 36, 60])
def test_a_large_column_that_nothing_reads(d_k, d_v, n, depth, exponent):
    """Column 5 of the state is 2^exponent times the others and no key or query has it, or the other way round: what is left of the
    32 columns around it carries the outputs."""
    for of_state in (True, False):
        prob = state_only(d_k, d_v, n, depth)
        big, none = ((prob.S0, (prob.q, prob.k)) if of_state else (prob.q, (prob.S0, prob.k)))
        for a in none:
            a[..., 5] = 0
        if of_state:
            big[..., 5] *= 2.0 ** exponent
            big[:, 1, :, : d_v // 2, 5] = 0.0                # rows without it, whole tiles of a sequence
        else:
            wide = synth.bf16_bits_to_f32(big[..., 5]) * np.float32(2.0 ** exponent)
            wide[:, ::3] = 0.0                               # nodes without it
            big[..., 5] = synth.f32_to_bf16_bits(wide)
        assert error_norm(prob, n) <= TOL_PRODUCTS, of_state


@pytest.mark.parametrize("d_k,d_v,n,depth", SHAPES)
def test_columns_of_every_magnitude(d_k, d_v, n, depth):
    """State and queries whose columns spread over 2^+-40 against each other, so that every one of them counts alike; some zero."""
    rng = np.random.default_rng(n)
    prob = state_only(d_k, d_v, n, depth)
    prob.k[:] = 0
    columns = 2.0 ** rng.integers(-40, 41, d_k)
    prob.S0 *= columns.astype(np.float32)
    prob.q[:] = synth.f32_to_bf16_bits((synth.bf16_bits_to_f32(prob.q) / columns).astype(np.float32))
    prob.S0[rng.random(prob.S0.shape) < 0.01] = 0.0
    assert error_norm(prob, n) <= TOL_PRODUCTS


@pytest.mark.parametrize("d_k,d_v,n,depth", SHAPES)
@pytest.mark.parametrize("state,query", [(112, 0), (118, 0), (118, -30), (-30, 118), (-60, 122), (-100, 0), (-60, -40), (60, 60)])
def test_results_inside_the_range_stay_inside(d_k, d_v, n, depth, state, query):
    """State and queries of 2^state and 2^query: the products are of 2^(state + query), and so are the outputs."""
    prob = state_only(d_k, d_v, n, depth)
    prob.S0 *= np.float32(2.0 ** state)
    prob.q[:] = synth.f32_to_bf16_bits((synth.bf16_bits_to_f32(prob.q) * np.float32(2.0 ** query)).astype(np.float32))
    assert error_norm(prob, n) <= TOL_PRODUCTS


@pytest.mark.parametrize("d_k,d_v,n,depth", SHAPES)
def test_values_of_tiles_that_are_done_again(d_k, d_v, n, depth):
    """The same large column with values beside the state, and one of these not finite: the nodes that have it on their path are
    not finite in that row, everything else is right."""
    rng = np.random.default_rng(n)
    trees = [synth.random_tree_parent(max(1, m), depth, 4, rng) for m in (n, n - 7)]
    prob = synth.make_problem(95 + n, 1, 3, d_k, d_v, trees, max_depth=depth, state_std=0.5)
    for a in (prob.q, prob.k):
        a[..., 5] = 0
    prob.S0[..., 5] *= 2.0 ** 40
    assert error_norm(prob, n) <= TOL_PRODUCTS
    ref = oracle_verify(prob)
    node, head, row = n // 2, 1, d_v - 1
    prob.v[0, node, head, row] = 0x7f80                              # infinity
    dp = DevProblem(prob, max_nodes=n)
    dp.verify_tree()
    assert dp.status_value() == 0
    o = dp.o.cpu().numpy().astype(np.float64)
    hit = np.zeros(o.shape, bool)
    hit[0, [t for t in range(n) if node in synth.root_path(trees[0], t)], head, row] = True
    assert not np.isfinite(o[hit]).any() and np.isfinite(o[~hit]).all()
    assert np.linalg.norm(o[~hit] - ref[~hit]) <= TOL_PRODUCTS * np.linalg.norm(ref[~hit])
