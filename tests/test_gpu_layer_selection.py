"""-m gpu: the selection of layers with more than 1024 candidates, layer by layer: next tokens, parents and counts of
layers_step against a selection in NumPy (n largest path values, lowest candidate index on ties, kept in index order) on the
device's own probabilities, so every bit is decided.  The logits of each layer are made for one way through the selection,
and the test checks that they take it."""
import math

import numpy as np
import pytest
import torch

from paper_2406_17276_b200 import binding, synth
from tests._gpu import poisoned_tree

pytestmark = pytest.mark.gpu


def _logits(kind, rows, V, k, rng):
    """bf16 bits [rows][V] of the nodes of a layer."""
    x = np.full((rows, V), -np.inf, np.float32)
    if kind == "ties":                                       # k tokens of 1/k each, exactly
        for r in range(rows):
            x[r, rng.choice(V, k, replace=False)] = 0.0
    elif kind == "narrow":                                   # everything within a few per cent of 1/V
        x = rng.integers(0, 9, (rows, V)).astype(np.float32) / 128.0
    elif kind == "spread":                                   # many factors of two, few candidates in each
        x = rng.normal(0.0, 3.0, (rows, V)).astype(np.float32)
    elif kind == "dense":                                    # a factor of two or so: many in each sixteenth of it
        for r in range(rows):
            x[r, rng.choice(V, k, replace=False)] = rng.uniform(-0.25, 0.25, k)
    else:                                                    # "crowded": what is kept comes from the first eighth of the nodes
        x = np.zeros((rows, V), np.float32)
        for r in range(max(1, rows // 8)):
            x[r] = -30.0
            x[r, rng.choice(V, k, replace=False)] = rng.uniform(-0.25, 0.25, k)
    return synth.f32_to_bf16_bits(x)


def _coarse(v):
    """Sixteen bins per factor of two, 1 at the top, everything below 2^-63 at the bottom; 1024 parts of each."""
    key = v.view(np.uint64) + 1
    e = (key >> np.uint64(48)).astype(np.int64) - (16 * 0x3FF - 1023)
    return np.clip(e, 0, 1023), ((key >> np.uint64(38)) & np.uint64(1023)).astype(np.int64)


def _way(v, n, survivors):
    """The way a layer of candidates v takes: one of listed / counted / split / digits (see select_layer_team_big)."""
    c, f = _coarse(v)
    nl = min(n, len(v))
    b = np.sort(c)[::-1][nl - 1]                             # the threshold's bin
    above, inside = c > b, c == b
    if above.sum() + inside.sum() > survivors and b > 0:
        s = np.sort(f[inside])[::-1][nl - above.sum() - 1]
        above, inside = above | (inside & (f > s)), inside & (f == s)
        split = True
    else:
        split = False
    kept = above | inside
    per = -(-(-(-len(v) // 4)) // 256) * 256
    if max(kept[q * per:(q + 1) * per].sum() for q in range(4)) > survivors // 4:
        return "digits"
    if split:
        return "split"
    return "counted" if inside.sum() > 64 and nl < kept.sum() else "listed"


@pytest.mark.parametrize("kind,n,k,D,want", [("ties", 64, 32, 14, "digits"), ("ties", 256, 16, 17, "digits"), ("ties", 300, 16, 6, "digits"),
                                             ("narrow", 256, 32, 4, "split"), ("narrow", 1024, 16, 5, "split"),
                                             ("spread", 256, 32, 6, "listed"), ("spread", 65, 16, 5, "listed"), ("spread", 1024, 32, 5, "listed"),
                                             ("dense", 64, 32, 5, "counted"), ("dense", 300, 16, 5, "counted"),
                                             ("crowded", 256, 32, 5, "digits"), ("crowded", 520, 32, 5, "digits")])
def test_selected_layers(kind, n, k, D, want):
    V, B = 512, 2
    rng = np.random.default_rng(n * 100 + k)
    ot = binding.OptTree(V, B * n, n, k, D, B)
    tree = poisoned_tree(ot, B)
    ot.layers_begin(B)
    cnt, phat = [1] * B, [np.ones(1)] * B
    ways, below = set(), False
    for d in range(1, D + 1):
        stride = max(cnt)
        x = _logits(kind, B * stride, V, k, rng)
        dev = torch.from_numpy(x.view(np.int16)).cuda()
        tok, prob = (t.cpu().numpy() for t in ot.row_softmax_topk(dev, torch.arange(B * stride, dtype=torch.int32, device="cuda")))
        nt, npar, nc = (t.cpu().numpy() for t in ot.layers_step(dev.view(B, stride, V), -math.inf, tree))
        for b in range(B):
            if d == D:
                assert nc[b] == 0
                continue
            at = slice(b * stride, b * stride + cnt[b])
            v = (phat[b][:, None] * prob[at]).ravel()
            N, nl = len(v), min(n, len(v))
            keep = np.sort(np.lexsort((np.arange(N), -v))[:nl])
            if N > 1024:
                ways.add(_way(v, n, 2048 if n > 256 else 1024))
                below = below or np.sort(v)[::-1][nl - 1] < 2.0 ** -63
            assert nc[b] == nl
            assert np.array_equal(nt[b, :nl], tok[at].ravel()[keep]), d
            assert np.array_equal(npar[b, :nl], keep // k), d
            cnt[b], phat[b] = nl, v[keep]
    assert ot.device_status() == 0
    assert want in ways, ways
    assert below == (kind == "ties" and n <= 256)            # the long ones reach thresholds below 2^-63
