"""-m gpu: verification of a tree whose node count is larger than the context's node budget: reported, and taken as full."""
import numpy as np
import pytest
import torch

from paper_2406_17276_b200 import binding, synth
from tests._gpu import dev_table

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,B,V", [(10, 3, 512), (256, 2, 1001), (1024, 1, 2048)])
def test_count_beyond_the_budget(n, B, V):
    H, k, D = 64, 16, 6
    ld = synth.draft_table(V, 3.0, 1.1, 5, H=H)
    ot = binding.OptTree(V, H, n, k, D, B)
    d = dev_table(ld)
    r = torch.from_numpy(synth.root_tokens(B, V, 3)).cuda()
    tree = ot.build(d, r, -np.inf)
    assert tree.n_sel.tolist() == [n] * B
    calls = [lambda: ot.verify(tree, d, r), lambda: ot.verify_sampled(tree, d, r, 1.0, 3, 4)]
    want = [[x.clone() for x in f()] for f in calls]
    assert ot.device_status() == 0
    tree.n_sel += torch.tensor([5000, 1, 77], dtype=torch.int32, device="cuda")[:B]
    for f, w in zip(calls, want):
        for _ in range(2):
            got = f()
            assert ot.device_status() == -5                  # OPT_TREE_ERR_INTERNAL
            assert all(torch.equal(a, b) for a, b in zip(got, w))
