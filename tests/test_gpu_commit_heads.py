"""Commit of two neighbouring 64 x 64 heads by one CTA, in large calls: bit for bit what the same sequences get in small calls, a
layer at a time, where a CTA has one head."""
import numpy as np
import pytest
import torch

from paper_2607_16673_b200 import binding as speca
from paper_2607_16673_b200 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rule", [0, speca.RULE_GATED_NO_ERASE])
@pytest.mark.parametrize("L,B,H", [(25, 20, 12), (26, 19, 13), (32, 16, 16)])
def test_large_calls_equal_small_ones(L, B, H, rule):
    rng = np.random.default_rng(L + B + H)
    n, depth = 16, 16
    offs = (np.arange(B + 1) * n).astype(np.int32)
    parent = np.tile(np.arange(-1, n - 1), B).astype(np.int32)
    T = B * n
    plen = rng.integers(0, depth + 1, B).astype(np.int32)
    plen[:3] = [0, 1, 16]
    pidx = np.tile(np.arange(depth), (B, 1)).astype(np.int32)
    pidx[4, 2] = 9                                    # not the parent's child: refused, left alone
    plen[4] = 5
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    S = synth.device_state(3, L, B, H, 64, 64, 0.5, "cuda")
    _, k, v, alpha, beta = synth.device_records(4, L, T, H, 64, 64, "cuda")
    args = (t(offs), T, t(parent), t(pidx), t(plen))
    whole, parts = S.clone(), S.clone()
    status, small = torch.zeros(1, dtype=torch.int32, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")
    speca.commit(speca.Dims(L, B, H, 64, 64, 1.0, depth, n, speca.ROUTE_AUTO, rule), whole, k, v, alpha, beta, *args, status)
    for l in range(L):
        one = speca.Dims(1, B, H, 64, 64, 1.0, depth, n, speca.ROUTE_AUTO, rule)
        speca.commit(one, parts[l:l + 1], k[l:l + 1], v[l:l + 1], alpha[l:l + 1], beta[l:l + 1], *args, small)
    assert int(status.item()) == int(small.item()) == speca.STATUS_BAD_PATH
    assert torch.equal(whole, parts)
    assert torch.equal(whole[:, 4], S[:, 4]) and torch.equal(whole[:, 0], S[:, 0]) and not torch.equal(whole[:, 2], S[:, 2])
