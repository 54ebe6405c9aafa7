"""-m gpu: whole builds (persistent, pruned, layer by layer) on aligned rows of more than two chunks (16384 logits), on either side of
where the builds begin to use the maxima of chunks (more than 32 pairs of a chunk and a winner, up to 32 chunks), against the oracle."""
import math

import numpy as np
import pytest
import torch

from paper_2406_17276_b200 import binding, synth
from tests import _compare
from tests._gpu import dev_table, poisoned_tree, tree_dict

pytestmark = pytest.mark.gpu
FIELDS = ("token", "parent", "depth", "phat", "n_sel", "depth_reached", "expected_len", "esub_trace")


@pytest.mark.parametrize("V,n,k,D,B,H", [(32776, 24, 10, 4, 2, 32), (32776, 24, 11, 4, 2, 32), (65536, 40, 8, 4, 2, 32), (65536, 300, 9, 4, 1, 32),
                                         (180224, 24, 8, 3, 2, 16), (524288, 8, 5, 2, 1, 8), (524296, 8, 5, 2, 1, 8)])
@pytest.mark.parametrize("delta", [-math.inf, 0.1])
def test_builds(V, n, k, D, B, H, delta):
    w = synth.Workload("long rows", B, V, n, k, D, 3.0, 1.1, 0.3, H=H, seed=V + n)
    ld, lt = synth.make_tables(w)
    table = dev_table(ld)
    ot = binding.OptTree(V, H, n, k, D, B)
    roots = synth.root_tokens(B, V, 5)
    r = torch.from_numpy(roots).cuda()
    full = ot.build(table, r, delta, poisoned_tree(ot, B))
    pruned, _ = ot.build_pruned(table, r, delta, poisoned_tree(ot, B))
    layered = poisoned_tree(ot, B)
    ot.layers_begin(B)
    toks, stride = r.view(-1, 1).to(torch.int64), 1
    for depth in range(D):
        rows = (toks[:, :stride].clamp(0, V - 1) * 31 + depth) % H
        nt, _, cnt = ot.layers_step(table[rows.reshape(-1)].view(B, stride, V).contiguous(), delta, layered)
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
