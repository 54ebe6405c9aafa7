"""-m gpu: steps of the layer-by-layer build that are not asked of the whole batch, or whose buffer is too narrow: every
sequence goes on from where it stands and ends with the tree of the persistent build."""
import math

import numpy as np
import pytest
import torch

from paper_2406_17276_b200 import binding, synth
from tests._gpu import dev_table, poisoned_tree

pytestmark = pytest.mark.gpu
FIELDS = ("token", "parent", "depth", "phat", "n_sel", "depth_reached", "expected_len", "esub_trace")
H, V, n, k, D, B = 64, 512, 12, 4, 6, 8


class _Driver:
    """Plays the draft model: keeps every sequence's next tokens and its own depth."""

    def __init__(self, delta, seed=3):
        self.d_ld = dev_table(synth.draft_table(V, 3.0, 1.1, 11, H=H))
        self.ot = binding.OptTree(V, H, n, k, D, B)
        self.delta = delta
        self.r = torch.from_numpy(synth.root_tokens(B, V, seed)).cuda()
        self.want = self.ot.build(self.d_ld, self.r, delta)
        self.tree = poisoned_tree(self.ot, B)
        self.ot.layers_begin(B)
        self.toks = [self.r[b:b + 1].to(torch.int64) for b in range(B)]
        self.depth = [0] * B

    def step(self, nb, stride=None):
        """One step of the first nb sequences; returns their counts."""
        stride = stride or max(1, max(len(t) for t in self.toks[:nb]))
        logits = torch.full((nb, stride, V), 0x7F00, dtype=torch.int16, device="cuda")      # huge logits beyond the counts
        for b in range(nb):
            rows = ((self.toks[b] * 31 + self.depth[b]) % H)[:stride]
            logits[b, :len(rows)] = self.d_ld[rows].view(torch.int16)
        nt, _, cnt = self.ot.layers_step(logits, self.delta, self.tree)
        cnt = cnt.cpu().tolist()
        for b in range(nb):
            if len(self.toks[b]) <= stride and len(self.toks[b]) > 0:
                self.toks[b] = nt[b, :cnt[b]].to(torch.int64)
                self.depth[b] += 1
        return cnt

    def check(self):
        torch.cuda.synchronize()
        assert self.ot.device_status() == 0
        assert all(len(t) == 0 for t in self.toks)
        for f in FIELDS:
            a, b = getattr(self.want, f).cpu().numpy(), getattr(self.tree, f).cpu().numpy()
            assert np.array_equal(a, b, equal_nan=True), f


@pytest.mark.parametrize("delta", [-math.inf, 0.25])
@pytest.mark.parametrize("calls", [[4, 8, 4, 8], [1, 8, 8, 3], [8, 2, 2, 2, 2, 2, 2, 8], [8, 7, 6, 5, 4, 3, 2, 1]])
def test_steps_of_fewer_sequences(calls, delta):
    g = _Driver(delta)
    for nb in calls + [B] * (2 * D):
        g.step(nb)
        if not any(len(t) for t in g.toks):
            break
    g.step(B)                                                # finished trees stay finished
    g.check()


@pytest.mark.parametrize("delta", [-math.inf, 0.25])
def test_a_buffer_too_narrow_for_a_layer_can_be_made_wider(delta):
    g = _Driver(delta)
    g.step(B)
    assert all(len(t) == k for t in g.toks)                  # layer 1: k nodes each
    assert g.step(B, stride=k - 1) == [0] * B                # no sequence can be grown from that
    assert g.ot.device_status() == -5                        # OPT_TREE_ERR_INTERNAL
    for _ in range(D):
        if any(len(t) for t in g.toks):
            g.step(B)
    g.check()
