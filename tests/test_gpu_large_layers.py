"""-m gpu: trees whose layers have more candidates than the layer team stages in shared memory (over 1024), against the oracle
and the pruned build.  Deep layers hardly reach a tree of ties or narrow distributions; which nodes their selection keeps is
checked in test_gpu_layer_selection.py."""
import math

import numpy as np
import pytest
import torch

from paper_2406_17276_b200 import binding, synth
from tests import _compare
from tests._gpu import dev_table, gpu_step

pytestmark = pytest.mark.gpu
FIELDS = ("token", "parent", "depth", "phat", "n_sel", "depth_reached", "expected_len", "esub_trace")


def _table(kind, H, V, k, rng):
    if kind == "peaked":
        return synth.draft_table(V, 3.0, 1.1, 11, H=H)
    if kind == "narrow":                                    # all probabilities within a few per cent of 1/V
        return synth.f32_to_bf16_bits((rng.integers(0, 9, (H, V)) / 128.0).astype(np.float32))
    ld = np.full((H, V), 0xFF80, np.uint16)                 # "ties": k tokens of logit 0 (terms that are powers of two: exact sums)
    for h in range(H):
        ld[h, rng.choice(V, k, replace=False)] = 0x0000
    return ld


@pytest.mark.parametrize("kind", ["peaked", "narrow", "ties"])
@pytest.mark.parametrize("n,k,D,B", [(64, 16, 5, 2), (65, 16, 5, 2), (130, 8, 6, 3), (256, 32, 5, 2), (257, 8, 6, 2), (512, 32, 4, 1), (1024, 32, 4, 1)])
def test_large_layers(kind, n, k, D, B):
    H, V = 64, 2048
    w = synth.Workload("large_layers", B, V, n, k, D, 3.0, 1.1, 0.0, H=H, seed=n + k)
    ld = _table(kind, H, V, k, np.random.default_rng(n * k))
    ot = binding.OptTree(V, H, n, k, D, B)
    d = dev_table(ld)
    roots = synth.root_tokens(B, V, 3)
    for delta in (-math.inf, 0.05):
        g = gpu_step(ot, d, d, roots, delta)
        if kind != "narrow":                                # (its path values tie within rounding)
            _o, st = _compare.compare_step(w, ld, ld, roots, delta, g)
            assert st["exact"] == B or kind == "peaked", st
        # the pruned build takes its own way through the selections and must agree bit for bit
        tree, _ = ot.build_pruned(d, torch.from_numpy(roots).cuda(), delta)
        torch.cuda.synchronize()
        for f in FIELDS:
            assert np.array_equal(g[f], getattr(tree, f).cpu().numpy()), f
    assert ot.device_status() == 0
