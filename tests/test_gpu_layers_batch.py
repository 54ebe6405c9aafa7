"""-m gpu: the layer-by-layer build where many sequences share a CTA's layer team: more sequences than CTAs, sequences that
stop at different layers, a buffer wider than the counts, and two batches one after the other in one context."""
import math

import numpy as np
import pytest
import torch

from paper_2406_17276_b200 import binding, synth
from tests._gpu import dev_table, poisoned_tree

pytestmark = pytest.mark.gpu
FIELDS = ("token", "parent", "depth", "phat", "n_sel", "depth_reached", "expected_len", "esub_trace")


def _layers(ot, d_ld, H, V, r, delta, D, wide):
    B = r.shape[0]
    tree = poisoned_tree(ot, B)
    ot.layers_begin(B)
    toks, cnt = r.view(-1, 1).to(torch.int64), torch.ones(B, dtype=torch.int32, device="cuda")
    for depth in range(D + 1):
        if int(cnt.max()) == 0:
            return tree
        stride = ot.cfg.n if wide and depth else max(1, int(cnt.max()))
        rows = ((toks[:, :stride].clamp(0, V - 1) * 31 + depth) % H).clamp_(0, H - 1)
        nt, _, cnt = ot.layers_step(d_ld[rows.reshape(-1)].reshape(B, stride, V).contiguous(), delta, tree)
        toks = nt.to(torch.int64)
    raise AssertionError("a tree did not stop by the depth limit")


@pytest.mark.parametrize("n,k,D,B,V,wide", [(8, 4, 4, 300, 512, False), (6, 3, 5, 700, 256, True), (1, 1, 3, 40, 64, False),
                                            (300, 8, 4, 9, 1024, True), (12, 3, 12, 64, 40960, False)])
@pytest.mark.parametrize("delta", [-math.inf, 0.25])
def test_same_trees_as_the_persistent_build(n, k, D, B, V, wide, delta):
    H = 64
    ld = synth.draft_table(V, 3.0, 1.1, n + k, H=H)
    d_ld = dev_table(ld)
    ot = binding.OptTree(V, H, n, k, D, B)
    for seed in (1, 2):                                      # the second batch meets the first one's leftovers
        r = torch.from_numpy(synth.root_tokens(B, V, seed)).cuda()
        got = _layers(ot, d_ld, H, V, r, delta, D, wide)
        want = ot.build(d_ld, r, delta, poisoned_tree(ot, B))
        torch.cuda.synchronize()
        assert ot.device_status() == 0
        for f in FIELDS:
            assert np.array_equal(getattr(want, f).cpu().numpy(), getattr(got, f).cpu().numpy(), equal_nan=True), f
