"""-m gpu: the selections whose keys the layer team holds in registers (layers of up to 1024 candidates, running top-n of up to 512
nodes), at the sizes where the held keys change in number and for both ways to the threshold (a listed bin, a bin too full for the
list): every layer's nodes and the final tree against a selection in NumPy on the device's own probabilities."""
import math

import numpy as np
import pytest
import torch

from paper_2406_17276_b200 import binding
from tests._gpu import dev_table, poisoned_tree, tree_dict
from tests.test_gpu_layer_selection import _coarse, _logits

pytestmark = pytest.mark.gpu


def _full_bin(v, n):
    """Whether the bin of the threshold holds more keys than the list (64) and not all of them are kept."""
    c = _coarse(v)[0]
    b = np.sort(c)[::-1][n - 1]
    return (c == b).sum() > 64 and (c >= b).sum() > n


@pytest.mark.parametrize("kind,n,k,D,full", [("spread", 8, 16, 6, False), ("spread", 43, 3, 6, False), ("spread", 32, 16, 6, False),
                                             ("spread", 27, 19, 5, False), ("spread", 33, 31, 5, False), ("spread", 64, 16, 7, False),
                                             ("spread", 256, 4, 7, False), ("spread", 257, 3, 7, False), ("spread", 512, 2, 12, False),
                                             ("ties", 64, 16, 5, True), ("ties", 20, 32, 14, True), ("ties", 256, 4, 7, True),
                                             ("narrow", 50, 10, 5, True), ("dense", 32, 32, 4, True), ("crowded", 40, 25, 4, True)])
def test_selected_layers_and_tree(kind, n, k, D, full):
    V, B = 512, 2
    rng = np.random.default_rng(n * 100 + k)
    ot = binding.OptTree(V, B * n, n, k, D, B)
    tree = poisoned_tree(ot, B)
    ot.layers_begin(B)
    cnt, phat, seen = [1] * B, [np.ones(1)] * B, False
    drafted = [[] for _ in range(B)]                         # per layer: values, tokens
    for d in range(1, D + 1):
        stride = max(cnt)
        dev = dev_table(_logits(kind, B * stride, V, k, rng))
        tok, prob = (t.cpu().numpy() for t in ot.row_softmax_topk(dev, torch.arange(B * stride, dtype=torch.int32, device="cuda")))
        nt, npar, nc = (t.cpu().numpy() for t in ot.layers_step(dev.view(B, stride, V), -math.inf, tree))
        for b in range(B):
            at = slice(b * stride, b * stride + cnt[b])
            v = (phat[b][:, None] * prob[at]).ravel()
            N, nl = len(v), min(n, len(v))
            seen = seen or (nl < N and _full_bin(v, nl))
            keep = np.sort(np.lexsort((np.arange(N), -v))[:nl])
            drafted[b].append((v[keep], tok[at].ravel()[keep]))
            assert nc[b] == (nl if d < D else 0)
            if d < D:
                assert np.array_equal(nt[b, :nl], tok[at].ravel()[keep]), d
                assert np.array_equal(npar[b, :nl], keep // k), d
            cnt[b], phat[b] = nl, v[keep]
    t = tree_dict(tree)
    for b in range(B):
        v, tk = (np.concatenate([layer[i] for layer in drafted[b]]) for i in (0, 1))
        keep = np.sort(np.lexsort((np.arange(len(v)), -v))[:n])
        assert t["n_sel"][b] == len(keep)
        assert np.array_equal(t["phat"][b, :len(keep)], v[keep]) and np.array_equal(t["token"][b, :len(keep)], tk[keep])
    assert ot.device_status() == 0
    assert seen == full


@pytest.mark.parametrize("kind,n,k", [("ties", 20, 32), ("ties", 64, 16), ("spread", 32, 16), ("narrow", 27, 19), ("crowded", 40, 25), ("spread", 256, 4)])
@pytest.mark.parametrize("delta", [-math.inf, -1.0])
def test_one_selection_or_two(kind, n, k, delta):
    """The pruned draft (one selection over the running top-n and the candidates, its rows sent out by it when there is no threshold)
    against the full one (a selection of each), equal path values included."""
    V, H, B, D = 512, 96, 5, 9
    d_ld = dev_table(_logits(kind, H, V, k, np.random.default_rng(n + k)))
    root = torch.arange(B, dtype=torch.int32, device="cuda") * 7
    ot = binding.OptTree(V, H, n, k, D, B)
    got = []
    for build in (ot.build, ot.build_pruned):
        tree = poisoned_tree(ot, B)
        build(d_ld, root, delta, tree)
        assert ot.device_status() == 0
        got.append(tree_dict(tree))
    for f in got[0]:
        assert np.array_equal(got[0][f], got[1][f]), f
