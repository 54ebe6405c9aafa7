"""-m gpu: draws of the verification with sampling that fall close to a running sum, on rows that are not 16-byte aligned
(double precision throughout) and at the largest rows of the one-pass path."""
import numpy as np
import pytest
import torch

import oracle
from paper_2406_17276_b200 import binding, synth
from tests._gpu import dev_table

pytestmark = pytest.mark.gpu
# u*S and the running sums are sums of up to V terms in double precision on both sides, each term good to a few 1e-16:
# relative to S they differ by far less than this
EXACT = 1e-11


def _shifted(tab, shift):
    """The table on the device, its first logit `shift` halves beyond a 256-byte boundary."""
    buf = torch.full((tab.size + 16,), 0x7F7F, dtype=torch.int16, device="cuda")
    buf[shift:shift + tab.size] = torch.from_numpy(tab.view(np.int16).reshape(-1)).cuda()
    return buf[shift:]


def _two_level_table(H, V, seed):
    """Every row one value up to a random place and another one from there on: a token's probability is everywhere about 1/V, and
    an approximate exponential errs the same way on every term of a stretch, which moves the running sums the most."""
    rng = np.random.default_rng(seed)
    x = np.empty((H, V), np.float32)
    for h in range(H):
        cut = int(rng.integers(V // 4, 3 * V // 4))
        x[h, :cut], x[h, cut:] = rng.integers(-255, 256, 2) / 256.0
    return synth.f32_to_bf16_bits(x)


def _draws(V, shift, B, steps, tau, margin, H=16):
    n, D = 1, 1
    lt = _two_level_table(H, V, V)
    ot = binding.OptTree(V, H, n, 1, D, B)
    target = _shifted(lt, shift)
    roots = np.arange(B, dtype=np.int32) * 7 % V
    r = torch.from_numpy(roots).cuda()
    tree = ot.build(dev_table(lt), r, -np.inf)
    t = [x.cpu().numpy() for x in (tree.token, tree.parent, tree.depth, tree.n_sel)]
    close, got = 0, []
    for step in range(steps):
        out = [x.cpu().numpy() for x in ot.verify_sampled(tree, target, r, tau, 99, step)]
        got.append(out)
        o = oracle.table_verify_sampled(lt, roots, *t, D, tau, 99, step)
        for b in range(B):
            same = all(np.array_equal(g[b], o[f][b]) for g, f in zip(out, ("accept_len", "accept_tokens", "accept_nodes", "next_root")))
            assert same or o["min_margin"][b] < margin, (step, b, o["min_margin"][b])
            close += EXACT < o["min_margin"][b] < 1e-7
    assert ot.device_status() == 0
    return got, close


@pytest.mark.parametrize("tau", [1.0, 0.25])
def test_unaligned_rows_draw_in_double_precision(tau):
    _, close = _draws(32003, 0, 64, 60, tau, EXACT)
    assert close > 0                                         # draws that single-precision sums would get wrong are among them


def test_draws_do_not_depend_on_the_address():
    want, _ = _draws(8004, 1, 64, 6, 1.0, EXACT)
    for shift in (2, 3, 4, 6, 7):
        got, _ = _draws(8004, shift, 64, 6, 1.0, EXACT)
        for a, b in zip(want, got):
            assert all(np.array_equal(x, y) for x, y in zip(a, b)), shift


# 640 segments of 512 logits take the one-pass path, longer rows the plain one
@pytest.mark.parametrize("V,margin", [(326664, 2e-6), (327680, 2e-6), (327688, EXACT), (327679, EXACT), (327681, EXACT)])
def test_largest_rows_of_the_one_pass_path(V, margin):
    _draws(V, 0, 4, 2, 1.0, margin, H=4)
