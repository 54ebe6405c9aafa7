"""-m gpu: whole builds (persistent, pruned, layer by layer) on rows that do not start on a 16-byte boundary, of several
chunks (16384 logits) and with both layouts of the layer scratch, against the oracle; the memory around the tables is
poisoned with the largest finite logits."""
import math

import numpy as np
import pytest
import torch

from paper_2406_17276_b200 import binding, synth
from tests import _compare
from tests._gpu import poisoned_tree, tree_dict

pytestmark = pytest.mark.gpu
FIELDS = ("token", "parent", "depth", "phat", "n_sel", "depth_reached", "expected_len", "esub_trace")


def _poisoned(size, shift):
    """`size` halves on the device, `shift` halves beyond a 256-byte boundary, with poison on either side."""
    buf = torch.full((size + 32,), 0x7F7F, dtype=torch.int16, device="cuda")
    return buf[8 + shift:8 + shift + size]


@pytest.mark.parametrize("V,n,k,D,B", [(16391, 24, 8, 5, 3), (33013, 24, 8, 5, 3), (33013, 300, 17, 4, 2), (49153, 48, 32, 4, 2)])
@pytest.mark.parametrize("shift", [1, 6])
@pytest.mark.parametrize("delta", [-math.inf, 0.1])
def test_builds(V, n, k, D, B, shift, delta):
    H = 32
    w = synth.Workload("unaligned", B, V, n, k, D, 3.0, 1.1, 0.3, H=H, seed=V + n)
    ld, lt = synth.make_tables(w)
    d_ld = _poisoned(ld.size, shift)
    d_ld.copy_(torch.from_numpy(ld.view(np.int16).reshape(-1)))
    assert d_ld.data_ptr() % 16 != 0
    ot = binding.OptTree(V, H, n, k, D, B)
    roots = synth.root_tokens(B, V, 5)
    r = torch.from_numpy(roots).cuda()
    full = ot.build(d_ld, r, delta, poisoned_tree(ot, B))
    pruned, _ = ot.build_pruned(d_ld, r, delta, poisoned_tree(ot, B))
    layered = poisoned_tree(ot, B)
    ot.layers_begin(B)
    toks, stride = r.view(-1, 1).to(torch.int64), 1
    table = torch.from_numpy(ld.view(np.int16)).cuda()
    for depth in range(D):
        rows = (toks[:, :stride].clamp(0, V - 1) * 31 + depth) % H
        buf = _poisoned(B * stride * V, shift).view(B, stride, V)
        buf.copy_(table[rows.reshape(-1)].view(B, stride, V))
        nt, _, cnt = ot.layers_step(buf, delta, layered)
        toks, stride = nt.to(torch.int64), max(1, int(cnt.max()))
    torch.cuda.synchronize()
    assert ot.device_status() == 0
    g = tree_dict(full)
    mask, pos = ot.mask(full, None)
    g.update(mask=mask.cpu().numpy(), position_ids=pos.cpu().numpy())
    _, st = _compare.compare_step(w, ld, lt, roots, delta, g, check_verify=False)
    assert st["exact"] == B, st
    for t in (pruned, layered):
        for f in FIELDS:
            assert np.array_equal(getattr(full, f).cpu().numpy(), getattr(t, f).cpu().numpy(), equal_nan=True), f
