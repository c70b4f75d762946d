"""Small-tree verification with rows, steps and nodes of very different magnitudes.  The products of larger trees work on fp16
pairs scaled by row of the state and by node, 32 columns at a time: a power of two on a row of the state and its values, or on a
query, must come out as that power of two and nothing else."""
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
