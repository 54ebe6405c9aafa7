"""-m gpu: the search for a long row's candidates (rows of more than two chunks of 16384 logits), which reads only the chunks in which
the consumers noted a maximum at or above the threshold, or, in rows with few chunks or few winners, all of a flagged thread's: at the
numbers of chunks and of pairs (flagged thread, chunk) where its way changes, on winners placed by hand, against a softmax and a sort in double precision."""
import numpy as np
import pytest
import torch

from paper_2406_17276_b200 import binding, synth
from tests._gpu import dev_table

pytestmark = pytest.mark.gpu
CHUNK, THREADS = 16384, 512


def _place(kind, V, k, rng):
    """Logits of one row."""
    if kind == "normal":
        return rng.normal(0.0, 3.0, V).astype(np.float32)
    x = rng.uniform(-30.0, -20.0, V).astype(np.float32)
    chunks = -(-V // CHUNK)
    if kind == "one_warp":                                   # a winner in every thread of one warp, all chunks taking part: 32 threads x chunks
        for t in range(32):
            c = t % chunks
            v = c * CHUNK + (96 + t) * 8 + t % 8
            x[min(v, V - 1)] = 1.0 + t / 64.0
    elif kind == "zeros":                                    # winners that are +0 and -0, the latter alone in their chunks and warps
        for i in range(k):
            x[((i % chunks) * CHUNK + (i * 37 % THREADS) * 8 + i % 8) % V] = 0.0 if i % 3 else -0.0
    else:                                                    # "last": the winners at the row's very end and start
        x[-(k - k // 2):] = np.linspace(2.0, 3.0, k - k // 2)
        x[:k // 2] = np.linspace(2.5, 3.5, k // 2)
    return x


@pytest.mark.parametrize("V,k", [(32776, 10), (49152, 2), (49153, 16), (81920, 5), (81928, 17), (128256, 16), (152063, 10), (163840, 32), (163848, 9), (180225, 32),
                                 (65536, 32), (65544, 12), (65544, 13), (81920, 12), (81920, 13),       # five chunks, 64 pairs of a chunk and a winner
                                 (200003, 10), (262144, 10), (262152, 3), (327688, 16),                 # maxima of several chunks kept together
                                 (524288, 5), (524296, 5), (524295, 4)])                                # 32 chunks, and one more
@pytest.mark.parametrize("kind", ["normal", "one_warp", "zeros", "last"])
def test_winners_of_long_rows(kind, V, k):
    H, rng = 3, np.random.default_rng(V + k)
    bits = synth.f32_to_bf16_bits(np.stack([_place(kind, V, k, rng) for _ in range(H)]))
    x = (bits.astype(np.uint32) << 16).view(np.float32).astype(np.float64)
    ot = binding.OptTree(V, H, k, k, 2, 1)
    tok, prob = (t.cpu().numpy() for t in ot.row_softmax_topk(dev_table(bits), torch.arange(H, dtype=torch.int32, device="cuda")))
    assert ot.device_status() == 0
    for r in range(H):
        want = np.lexsort((np.arange(V), -x[r]))[:k]         # (larger first, lower token on ties; -0 ties with +0)
        e = np.exp(x[r] - x[r].max())
        assert np.array_equal(tok[r], want)
        # single-precision terms, a few 1e-7 of the sum (the library's stated error of a probability)
        np.testing.assert_allclose(prob[r], e[want] / e.sum(), rtol=1e-6)
