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


@pytest.mark.parametrize("V", [1, 5, 9, 513, 4103, 33013])
@pytest.mark.parametrize("B", [1, 64, 130])                  # 9 rows take blocks of 512 threads, 576 of 256, 1170 of 128 (148 SMs)
@pytest.mark.parametrize("shift", [0, 1, 7])
def test_verification_at_any_offset(V, B, shift):
    n, k, D, H = 8, min(4, V), 5, 17
    ld, lt = _defs.small_table(H, V, V), _defs.small_table(H, V, V)
    lt[::3] = _defs.small_table(H, V, V + 1)[::3]            # the target disagrees on a third of the rows
    ot = binding.OptTree(V, H, n, k, D, B)
    roots = np.arange(B, dtype=np.int32) % V
    r = torch.from_numpy(roots).cuda()
    tree = ot.build(_at(ld, 0), r, -np.inf)
    target = _at(lt, shift)
    t = [x.cpu().numpy() for x in (tree.token, tree.parent, tree.depth, tree.n_sel)]
    got = [x.cpu().numpy() for x in ot.verify(tree, target, r)]
    for b in range(B):                                       # the walk, by definition
        cur, A, path = -1, 0, []
        while True:
            tok, dep = (roots[b], 0) if cur < 0 else (t[0][b, cur], t[2][b, cur])
            x, _ = _defs.np_row_probs(lt, tok, dep)
            y = int(_defs.np_topk(x, 1)[0])
            assert got[1][b, A] == y
            A += 1
            hit = [i for i in range(t[3][b]) if t[1][b, i] == cur and t[0][b, i] == y]
            if A > D or not hit:
                break
            cur = hit[0]
            path.append(cur)
        assert got[0][b] == A and got[3][b] == y
        assert got[1][b, A:].tolist() == [-1] * (D + 1 - A)
        assert got[2][b].tolist() == path + [-1] * (D - len(path))
    out = [x.cpu().numpy() for x in ot.verify_sampled(tree, target, r, 1.0, 77, 3)]
    o = oracle.table_verify_sampled(lt, roots, *t, D, 1.0, 77, 3)
    for b in range(B):
        same = all(np.array_equal(g[b], o[f][b]) for g, f in zip(out, ("accept_len", "accept_tokens", "accept_nodes", "next_root")))
        assert same or o["min_margin"][b] < 2e-6             # a draw that close to a running sum may fall either way
    assert ot.device_status() == 0
