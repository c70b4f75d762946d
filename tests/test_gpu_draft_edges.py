"""The integer kernels at the edges of their fast forms (sequences of up to 64 nodes pruned by a warp, masks of up to 64
nodes as words, up to 128 nodes staged for acceptance, rows of the convolution state in pieces): bit-exact."""
import numpy as np
import pytest
import torch

import oracle
from paper_2607_16673_b200 import binding as speca
from paper_2607_16673_b200 import synth

pytestmark = pytest.mark.gpu
t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
I32 = dict(dtype=torch.int32, device="cuda")


def pack(parents):
    offs = np.concatenate([[0], np.cumsum([len(p) for p in parents])]).astype(np.int32)
    return offs, np.concatenate(parents).astype(np.int32)


def prune(N, tau, budget, offs, parent, logp):
    T, B = len(parent), len(offs) - 1
    oo, op, oi, status = torch.full((B + 1,), -7, **I32), torch.full((T,), -7, **I32), torch.full((T,), -7, **I32), torch.zeros(1, **I32)
    speca.prune_tree(N, tau, budget, t(offs), t(parent), t(logp), oo, op, oi, status)
    return oo.cpu().numpy(), op.cpu().numpy(), oi.cpu().numpy(), int(status.item())


@pytest.mark.parametrize("B,N", [(1, 64), (2, 1), (9, 64), (127, 33), (128, 64), (129, 64), (20, 65)])
def test_pruning_of_small_batches(B, N):
    """Both forms around the line between them: chains of 64 levels, forests, empty sequences, ties, scores that rise."""
    rng = np.random.default_rng(400 + B + N)
    parents = [synth.random_tree_parent(int(n), min(N, 16), 4, rng) for n in rng.integers(1, N + 1, B)]
    parents[0] = synth.chain_parent(N)
    if B > 2:
        parents[1], parents[2] = np.full(N, -1, np.int32), np.zeros(0, np.int32)
    offs, parent = pack(parents)
    logp = np.log(rng.uniform(0.02, 1.5, len(parent))).astype(np.float32)
    logp[rng.random(len(parent)) < 0.3] = -0.5
    for tau, budget in ((0.0, 3), (2.0, N), (1e4, max(1, N // 3)), (1e4, 0)):
        oo, op, oi, status = prune(N, tau, budget, offs, parent, logp)
        ro, rp, ri = oracle.prune_tree(offs, parent, logp, tau, budget)
        n = int(ro[-1])
        assert status == 0 and np.array_equal(oo, ro)
        assert np.array_equal(op[:n], rp) and np.array_equal(oi[:n], ri) and np.all(op[n:] == -7) and np.all(oi[n:] == -7)


def test_pruning_reports_bad_sequences_and_keeps_nothing_of_them():
    """A parent that is no earlier node, a sequence over the limit: reported, no output; the others as if they were empty."""
    good = [synth.chain_parent(5), synth.chain_parent(9), synth.chain_parent(3)]
    for bad, code in ((np.array([-1, 1, 0], np.int32), speca.STATUS_BAD_PARENT), (synth.chain_parent(17), speca.STATUS_TOO_MANY)):
        offs, parent = pack([good[0], bad, good[1], good[2]])
        logp = -np.arange(1, len(parent) + 1, dtype=np.float32) / 64
        oo, op, oi, status = prune(16, 1e4, 16, offs, parent, logp)
        assert status == code and oo.tolist() == [0, 5, 5, 14, 17]
        assert op[:17].tolist() == [*range(-1, 4), *range(-1, 8), *range(-1, 2)]


def test_pruning_with_scores_that_are_no_numbers():
    """What the two forms do with values that are not finite is the same."""
    rng = np.random.default_rng(7)
    parents = [synth.random_tree_parent(40, 8, 4, rng) for _ in range(6)]
    offs, parent = pack(parents)
    logp = np.log(rng.uniform(0.02, 1.0, len(parent))).astype(np.float32)
    logp[offs[1]], logp[offs[2] + 7], logp[offs[3] + 3], logp[offs[4]] = np.nan, np.nan, -np.inf, -np.inf
    logp[offs[5] + 5] = np.inf
    for tau, budget in ((3.0, 12), (1e4, 20)):
        small, large = prune(64, tau, budget, offs, parent, logp), prune(65, tau, budget, offs, parent, logp)
        n = int(large[0][-1])
        assert np.array_equal(small[0], large[0]) and np.array_equal(small[1][:n], large[1][:n]) and np.array_equal(small[2][:n], large[2][:n])


@pytest.mark.parametrize("n", [1, 31, 32, 33, 64, 65, 128, 129, 256, 257])
def test_acceptance_at_the_limits_of_what_is_staged(n):
    """Greedy and stochastic acceptance of sequences of n nodes beside small ones, and what they refuse."""
    rng = np.random.default_rng(500 + n)
    parents = [synth.random_tree_parent(n, 8, 8, rng), synth.chain_parent(min(n, 8)), np.zeros(0, np.int32),
               synth.random_tree_parent(max(1, n - 1), 8, 6, rng), synth.chain_parent(2)]
    offs, parent = pack(parents)
    T, B = len(parent), len(parents)
    draft, target, root = rng.integers(0, 3, T), rng.integers(0, 3, T), rng.integers(0, 3, B)
    pd = rng.uniform(0.1, 1, T).astype(np.float32)
    pt, u = (pd * rng.uniform(0.4, 1.2, T)).astype(np.float32), rng.random(T).astype(np.float32)
    for bad in (False, True):
        if bad:
            parent = parent.copy()
            parent[offs[0] + n - 1] = n - 1              # its own parent: the sequence is refused, the others are not
        pidx, plen, nxt, status = torch.full((B, 8), -7, **I32), torch.full((B,), -7, **I32), torch.full((B,), -7, **I32), torch.zeros(1, **I32)
        i32 = lambda a: t(np.asarray(a, np.int32))
        speca.greedy_accept(B, 8, t(offs), t(parent), i32(draft), i32(target), i32(root), pidx, plen, nxt, status)
        sidx, slen, sstat = torch.full((B, 8), -7, **I32), torch.full((B,), -7, **I32), torch.zeros(1, **I32)
        speca.stochastic_accept(B, 8, t(offs), t(parent), t(pt), t(pd), t(u), sidx, slen, sstat)
        want = (oracle.greedy_accept(offs, pack(parents)[1], draft.astype(np.int32), target.astype(np.int32), root.astype(np.int32), 8),
                oracle.stochastic_accept(offs, pack(parents)[1], pt, pd, u, 8))
        skip = int(bad)
        assert int(status.item()) == int(sstat.item()) == (speca.STATUS_BAD_PARENT if bad else 0)
        if bad:
            for idx, ln in ((pidx, plen), (sidx, slen)):
                assert int(ln[0]) == 0 and idx[0].tolist() == [-1] * 8
            assert int(nxt[0]) == root[0]
        assert np.array_equal(pidx.cpu().numpy()[skip:], want[0][0][skip:]) and np.array_equal(plen.cpu().numpy()[skip:], want[0][1][skip:])
        assert np.array_equal(nxt.cpu().numpy()[skip:], want[0][2][skip:])
        assert np.array_equal(sidx.cpu().numpy()[skip:], want[1][0][skip:]) and np.array_equal(slen.cpu().numpy()[skip:], want[1][1][skip:])


@pytest.mark.parametrize("n", [1, 32, 33, 64, 65])
def test_masks_that_are_no_tree_masks_are_refused(n):
    """Self bit missing, a later node among the ancestors, an ancestor missing: refused in both forms, the neighbour is not."""
    rng = np.random.default_rng(600 + n)
    tree = synth.random_tree_parent(n, 8, 3, rng)
    offs, parent = pack([tree, tree])
    mask = np.zeros((2, n, n), np.uint8)
    for i in range(n):
        mask[:, i, synth.root_path(tree, i)] = 3                     # any byte but zero counts
    depth = synth.depth_of(tree)
    faults = [(n - 1, n - 1, 0)] + ([(0, n - 1, 1)] if n > 1 else [])
    if depth.max() >= 3:
        deep = int(np.argmax(depth))
        faults.append((deep, synth.root_path(tree, deep)[0], 0))
    for fault in [None] + faults:
        m = mask.copy()
        if fault:
            m[0, fault[0], fault[1]] = fault[2]
        got, status = torch.full((2 * n,), -7, **I32), torch.zeros(1, **I32)
        speca.tree_mask_to_parent(t(m), t(offs), got, status)
        assert int(status.item()) == (speca.STATUS_BAD_PARENT if fault else 0)
        assert np.array_equal(got.cpu().numpy(), np.concatenate([np.full(n, -7) if fault else tree, tree]))


@pytest.mark.parametrize("W,ch", [(4, 4088), (4, 4096), (5, 4104), (3, 8200)])
def test_convolution_rows_around_the_pieces_of_a_block(W, ch):
    rng = np.random.default_rng(W * ch)
    offs, L, T = np.array([0, 16, 17, 22], np.int32), 2, 22
    C, x = rng.integers(0, 65536, (L, 3, W, ch), dtype=np.uint16), rng.integers(0, 65536, (L, T, ch), dtype=np.uint16)
    pidx, plen = np.full((3, 16), -1, np.int32), np.array([16, 1, 0], np.int32)
    pidx[0], pidx[1, 0] = np.arange(16), 0
    dev = lambda a: t(a.view(np.int16)).view(torch.bfloat16)
    Cd, status = dev(C), torch.zeros(1, **I32)
    speca.commit_conv(Cd, dev(x), t(offs), T, t(pidx), t(plen), status)
    assert int(status.item()) == 0
    assert np.array_equal(Cd.view(torch.int16).cpu().numpy().view(np.uint16), oracle.commit_conv(C, x, offs, pidx, plen))
