"""-m gpu: builds repeated back to back, whose layers hand words from SM to SM at ever different moments, give the same bits
every time, and those of the layer-by-layer build, which a kernel's end orders."""
import math

import numpy as np
import pytest
import torch

from paper_2406_17276_b200 import binding, synth
from tests._gpu import dev_table, poisoned_tree

pytestmark = pytest.mark.gpu
FIELDS = ("token", "parent", "depth", "phat", "n_sel", "depth_reached", "expected_len", "esub_trace")


def _layers(ot, d_ld, H, V, r, delta, D):
    B = r.shape[0]
    tree = poisoned_tree(ot, B)
    ot.layers_begin(B)
    toks, cnt = r.view(-1, 1).to(torch.int64), torch.ones(B, dtype=torch.int32, device="cuda")
    for depth in range(D + 1):
        stride = int(cnt.max())
        if stride == 0:
            break
        rows = ((toks[:, :stride].clamp(0, V - 1) * 31 + depth) % H).clamp_(0, H - 1)
        nt, _, cnt = ot.layers_step(d_ld[rows.reshape(-1)].reshape(B, stride, V).contiguous(), delta, tree)
        toks = nt.to(torch.int64)
    return tree


# short rows (a layer's last words come in while the team is at work), layers of one and of several candidates per thread, of more than
# the shared memory holds, layer 1 by the finisher and by the team, more sequences than CTAs
@pytest.mark.parametrize("n,k,D,B,V", [(16, 8, 8, 1, 256), (40, 10, 10, 9, 512), (128, 16, 10, 3, 512), (200, 32, 8, 2, 1024),
                                       (512, 16, 7, 2, 512), (8, 16, 8, 4, 256), (12, 4, 6, 200, 256)])
@pytest.mark.parametrize("delta", [-math.inf, 0.02])
def test_repeated_builds(n, k, D, B, V, delta):
    H = 64
    d_ld = dev_table(synth.draft_table(V, 1.0, 1.1, n + k, H=H))
    ot = binding.OptTree(V, H, n, k, D, B)
    r = torch.from_numpy(synth.root_tokens(B, V, 3)).cuda()
    want = _layers(ot, d_ld, H, V, r, delta, D)
    full = [ot.build(d_ld, r, delta, poisoned_tree(ot, B)) for _ in range(60)]
    pruned = [ot.build_pruned(d_ld, r, delta, poisoned_tree(ot, B))[0] for _ in range(60)]
    torch.cuda.synchronize()
    assert ot.device_status() == 0
    for f in FIELDS:
        w = getattr(want, f).cpu().numpy()
        for t in full + pruned:
            assert np.array_equal(w, getattr(t, f).cpu().numpy(), equal_nan=True), f
