"""-m gpu: every kind of bounded device-side wait gives up with a timeout status instead of hanging.

opt_tree_selftest_waits enters each wait on something nobody completes (a fresh shared-memory barrier,
words that stay zero, a row source that never has a row) with a limit of microseconds; the kernel must
end and every wait must have recorded OPT_TREE_ERR_TIMEOUT in its own status word.  The context stays
usable afterwards.
"""
import math

import numpy as np
import pytest
import torch

from paper_2406_17276_b200 import binding, synth
from tests._gpu import dev_table

pytestmark = pytest.mark.gpu


def test_every_bounded_wait_runs_out_and_reports_a_timeout():
    w = synth.Workload("waits", 2, 512, 8, 4, 4, 3.0, 1.1, 0.3, H=16, seed=2)
    ld, _ = synth.make_tables(w)
    ot = binding.OptTree(w.V, w.H, w.n, w.k, w.max_depth, w.batch)
    res = ot.selftest_waits()
    torch.cuda.synchronize()
    assert res.cpu().tolist() == [binding.ERR_TIMEOUT] * 5
    assert ot.device_status() == 0                                   # the context's own word is untouched
    # the context still builds trees
    tree = ot.build(dev_table(ld), torch.from_numpy(synth.root_tokens(2, w.V, 1)).cuda(), -math.inf)
    torch.cuda.synchronize()
    assert ot.device_status() == 0 and int(tree.n_sel.min()) == w.n


@pytest.mark.parametrize("n,k,rows,written,joint", [
    (64, 10, 20, 3, False), (64, 10, 20, 0, False), (64, 10, 64, 2, False),          # candidates in registers, four or eight per thread
    (256, 16, 100, 5, False), (256, 16, 100, 0, False), (600, 16, 600, 10, False), (600, 16, 80, 0, False),      # large layers, both scratch layouts
    (64, 10, 20, 3, True), (64, 10, 40, 0, True), (64, 10, 64, 5, True), (600, 16, 60, 4, True),                 # with the running top-n
    (64, 10, 20, 20, False), (64, 10, 64, 64, False), (256, 16, 100, 100, False), (600, 16, 600, 600, False), (64, 10, 20, 20, True), (64, 10, 64, 64, True)])
def test_candidates_that_never_come_count_as_token_0_of_path_value_0_and_a_timeout_is_reported(n, k, rows, written, joint):
    V = 12007
    ot = binding.OptTree(V, 16, n, k, 3, 2)
    res, tok, par, ph = (x.cpu().numpy() for x in ot.selftest_selection(rows, written, joint))
    assert res.tolist() == [binding.OK if written == rows else binding.ERR_TIMEOUT]
    nl = min(rows * k, n - 1 if joint else n)              # (the one node of layer 1 has the largest path value and stays)
    i = np.arange(rows * k)
    there = i < written * k
    value = np.where(there, 0.5 ** (1 + i % 3), 0.0)
    kept = np.sort(np.lexsort((i, -value))[:nl])           # ties by lowest index, kept in index order
    np.testing.assert_array_equal(tok[:nl], np.where(there, i % V, 0)[kept])
    np.testing.assert_array_equal(par[:nl], kept // k)
    np.testing.assert_array_equal(ph[:nl], value[kept])
    assert (tok[nl:] == -1).all() and (par[nl:] == -1).all() and (ph[nl:] == -1).all()
    # the context still builds trees
    w = synth.Workload("waits", 2, V, n, k, 3, 3.0, 1.1, 0.3, H=16, seed=2)
    tree = ot.build(dev_table(synth.make_tables(w)[0]), torch.from_numpy(synth.root_tokens(2, V, 1)).cuda(), -math.inf)
    torch.cuda.synchronize()
    assert ot.device_status() == 0 and int(tree.n_sel.min()) == n
