"""A key or value that is not finite stays on the root paths it belongs to (Section 4.2: siblings never influence each
other), on the kernels that multiply whole blocks of nodes with zero weights off the path."""
import numpy as np
import pytest
import torch

from paper_2607_16673_b200 import binding as speca
from paper_2607_16673_b200 import synth
from gpu_util import DevProblem

pytestmark = pytest.mark.gpu

SHAPES = [  # L, B, H, d_k, d_v, nodes, depth, chain, route, with u
    (1, 3, 2, 64, 64, 8, 8, True, speca.ROUTE_AUTO, False),
    (1, 3, 2, 64, 96, 24, 6, False, speca.ROUTE_AUTO, False),
    (1, 3, 2, 64, 64, 61, 16, False, speca.ROUTE_AUTO, False),        # split between two warps
    (1, 3, 2, 128, 128, 13, 6, False, speca.ROUTE_AUTO, False),
    (1, 3, 2, 128, 256, 32, 8, False, speca.ROUTE_AUTO, False),
    (1, 3, 2, 256, 96, 30, 8, False, speca.ROUTE_AUTO, False),
    (1, 3, 2, 256, 256, 8, 8, True, speca.ROUTE_AUTO, False),
    (1, 3, 2, 128, 256, 16, 8, False, speca.ROUTE_EFFECTIVE, False),
    (1, 3, 2, 128, 256, 61, 8, False, speca.ROUTE_EFFECTIVE, False),  # both halves of the node set
    (1, 3, 2, 128, 128, 50, 16, False, speca.ROUTE_EFFECTIVE, True),
    (1, 3, 2, 256, 256, 30, 16, False, speca.ROUTE_EFFECTIVE, True),
    (4, 19, 16, 128, 256, 40, 8, False, speca.ROUTE_EFFECTIVE, False),  # the form for large calls
]


@pytest.mark.parametrize("value", [float("nan"), float("inf")])
@pytest.mark.parametrize("what", ["k", "v"])
@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "-".join(map(str, s)))
def test_a_value_that_is_not_finite_stays_on_its_paths(shape, what, value):
    L, B, H, dk, dv, n, depth, chain, route, with_u = shape
    rng = np.random.default_rng(n * dk + depth)
    parents = [synth.chain_parent(n) if chain else synth.random_tree_parent(n, depth, 4, rng) for _ in range(B)]
    prob = synth.make_problem(n, L, H, dk, dv, parents, max_depth=depth)
    p = DevProblem(prob, route, want_u=with_u)
    seq, nodes, head, col = 1, (n // 3, n - 2), 1, 5            # two nodes of the middle sequence, one head
    x = {"k": p.k, "v": p.v}[what]

    def verify(val):
        for t in nodes:
            x[0, seq * n + t, head, col] = val
        p.o.fill_(-7.0)
        (p.verify_chain if chain else p.verify_tree)()
        assert p.status_value() == 0
        return [r.clone() for r in (p.o, p.u) if r is not None]

    clean, dirty = verify(0.0), verify(value)
    hit = torch.zeros(p.T, dtype=torch.bool)
    for t in range(n):
        a = t
        while a >= 0:
            hit[seq * n + t] |= a in nodes
            a = int(parents[seq][a])
    assert 0 < int(hit.sum()) < n
    for c, d in zip(clean, dirty):
        touched = torch.zeros_like(c, dtype=torch.bool)
        touched[0, hit.to(c.device), head, col if what == "v" else slice(None)] = True
        assert torch.equal(c[~touched], d[~touched])            # zero weights: the same sums, bit for bit
        assert torch.isfinite(c).all()
        assert not torch.isfinite(d[touched]).any()


@pytest.mark.parametrize("route", [speca.ROUTE_AUTO, speca.ROUTE_EFFECTIVE])
def test_a_large_finite_key_is_not_taken_for_an_infinite_one(route):
    """The square of a key of 2^70 does not fit fp32, the key itself counts."""
    parents = [np.array([-1, 0, 0], np.int32)]
    prob = synth.make_problem(2, 1, 2, 128, 128, parents, max_depth=3)
    p = DevProblem(prob, route)
    p.k[0, 0, 0] *= 2.0 ** 70
    p.beta[0, 0, 0] = 2.0 ** -100
    p.verify_tree()
    ref = DevProblem(prob, speca.ROUTE_SERIAL)
    ref.k.copy_(p.k)
    ref.beta.copy_(p.beta)
    ref.verify_tree()
    assert p.status_value() == 0 and ref.status_value() == 0
    assert float(ref.o.abs().max()) > 2.0 ** 20
    # sums that cancel in powers of two: looser than fp32 rounding, a key left out would show at full size
    assert float((p.o - ref.o).abs().max()) < 1e-4 * float(ref.o.abs().max())
