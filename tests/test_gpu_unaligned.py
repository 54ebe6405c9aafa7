"""-m gpu: rows that do not start on a 16-byte boundary (a vocabulary that is no multiple of eight, an odd table
base), at the sizes where granules, vectors and chunks (16384 logits) end."""
import numpy as np
import pytest
import torch

import oracle
from paper_2406_17276_b200 import binding
from tests import _defs

pytestmark = pytest.mark.gpu


def _at(tab: np.ndarray, shift: int) -> torch.Tensor:
    """The table on the device, its first logit `shift` halves beyond a 256-byte boundary, poisoned around."""
    buf = torch.full((tab.size + 16,), 0x7F80 - 1, dtype=torch.int16, device="cuda")      # huge finite logits
    buf[shift:shift + tab.size] = torch.from_numpy(tab.view(np.int16).reshape(-1)).cuda()
    return buf[shift:]


@pytest.mark.parametrize("V,k", [(1, 1), (7, 3), (9, 9), (15, 10), (16383, 10), (16384, 10), (16385, 10), (16391, 32), (16400, 16),
                                 (32761, 10), (32771, 17), (50257, 10), (128257, 16)])
@pytest.mark.parametrize("shift", [0, 1, 6, 7])
def test_rows_at_any_offset(V, k, shift):
    H = 9                                                    # with an odd V the rows take all eight offsets
    tab = _defs.small_table(H, V, V + k)
    ot = binding.OptTree(V, H, 8, k, 4, 1)
    rows = torch.arange(H - 1, -1, -1, dtype=torch.int32, device="cuda")
    tok, prob = ot.row_softmax_topk(_at(tab, shift), rows)
    torch.cuda.synchronize()
    assert ot.device_status() == 0
    for i in range(H):
        etok, ep, _m, _S = oracle.row_softmax_topk(tab[H - 1 - i], k)
        assert tok[i].cpu().numpy().tolist() == etok.tolist()
        # single-precision terms and sums of a few thousand logits per thread: about 1e-7, ten times that allowed
        np.testing.assert_allclose(prob[i].cpu().numpy(), ep, rtol=2e-6)


def test_a_row_gives_the_same_bits_at_every_offset():
    V, k, H = 32000, 10, 3
    tab = _defs.small_table(H, V, 5)
    ot = binding.OptTree(V, H, 8, k, 4, 1)
    rows = torch.arange(H, dtype=torch.int32, device="cuda")
    want = ot.row_softmax_topk(_at(tab, 0), rows)
    for shift in range(1, 8):
        got = ot.row_softmax_topk(_at(tab, shift), rows)
        assert torch.equal(want[0], got[0]) and torch.equal(want[1], got[1]), shift
    assert ot.device_status() == 0
