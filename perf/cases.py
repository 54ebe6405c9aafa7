"""Performance cases of the OPT-Tree library: what a decoding loop asks of it, through its public binding.

A decoding step hands the library two sets of logits that are already on the GPU (the draft model's and the target
model's, here tables of the recipe in paper_2406_17276_b200/synth.py, drawn on the device) and the last accepted token of every
sequence, and takes the tree, its attention mask and the accepted tokens.  The forms in which that happens (`op`):

  step      build -> mask -> verify, everything on the device: the ordinary step of a serving loop
  pruned    build_pruned -> mask -> verify -> post_verify: the same trees from the rows that still matter, with the dense mask and
            the cache keep list that the target forward and the caches consume
  sampled   build with a threshold -> mask -> verify_sampled at temperature 1
  layers    layers_begin, then one layers_step per drafted layer with the logits of that layer's nodes: the form for a real draft model
  rows      row_softmax_topk over a list of rows: the draft step of callers that keep their own trees
  host      step_host: root tokens from host memory, every result back in host memory

Sizes are those of synth.WORKLOADS and of the tests (node budgets 10 ... 512, vocabularies 32000 ... 152064, batches 1 ... 64), and
vocabularies that are no multiple of eight, whose rows are not 16-byte aligned.
"""
import math

import torch

from paper_2406_17276_b200 import binding, synth

H = synth.H_ROWS
OFF = -math.inf


def listed():
    def case(name, op, B, V, n, k, D, sigma=3.0, s=1.1, q=0.2, delta="off", rows=0):
        return dict(name=name, op=op, B=B, V=V, n=n, k=k, D=D, sigma=sigma, s=s, q=q, delta=delta, rows=rows)
    return [
        case("step-b1-n10", "step", 1, 32000, 10, 10, 6),                        # one user, the smallest budget: latency
        case("step-b1-n50", "step", 1, 32000, 50, 10, 10, 4.0, 1.3, 0.1),        # one user, the paper's usual budget
        case("step-b1-wide", "step", 1, 128256, 64, 16, 12),                     # one user, a wide vocabulary
        case("step-b32", "step", 32, 32000, 64, 10, 10),                         # a serving batch: the benchmark's workload
        case("step-b64-n256-wide", "step", 64, 152064, 256, 32, 20, 2.5, 1.05),  # the largest: batch, budget and vocabulary
        case("step-b16-ragged", "step", 16, 32003, 48, 8, 8),                    # a vocabulary with added tokens: unaligned rows
        case("step-b2-n512", "step", 2, 32000, 512, 16, 12),                     # the large trees of the budget sweep
        case("pruned-b32", "pruned", 32, 32000, 64, 10, 10),                     # the serving batch from the rows that still matter
        case("sampled-b8-delta", "sampled", 8, 32000, 60, 10, 10, delta=0.2),    # growth stopped by the threshold, temperature 1
        case("layers-b8", "layers", 8, 32000, 50, 10, 10),                       # a real draft model between the layers
        case("rows-ragged", "rows", 1, 50257, 8, 10, 4, rows=1999),              # the row step alone, unaligned rows
        case("host-b32", "host", 32, 32000, 64, 10, 10),                         # the serving batch with host buffers
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["step", "step", "step", "pruned", "sampled", "layers", "rows", "host"])
    V = _log_int(rng, 8000, 152064)
    if rng.random() < 0.6:
        V = V // 8 * 8
    c = dict(op=op, B=_log_int(rng, 1, 64), V=V, n=_log_int(rng, 10, 512), k=rng.randint(4, 32), D=rng.randint(4, 20),
             sigma=rng.choice([2.5, 3.0, 4.0]), s=rng.choice([1.05, 1.1, 1.3]), q=rng.choice([0.1, 0.2]), delta="off", rows=0)
    if op == "sampled":
        c["delta"] = rng.choice([0.0, 0.2, 0.5])
    if op == "rows":
        c.update(B=1, n=8, D=4, rows=_log_int(rng, 16, 20000))
    if op == "layers":                                      # its logits are all held at once: 2 GB at most
        while _rows(c) * V > 1 << 30:
            c["n"], c["B"] = max(10, c["n"] // 2), max(1, c["B"] // 2)
    # at most half of the largest listed case; unaligned rows, which have cost fifty times an aligned one, at most a hundredth
    most = 297024 * 152064 // (2 if V % 8 == 0 else 100)
    while _rows(c) * V > most:
        if c["op"] == "rows":
            c["rows"] //= 2
        elif c["B"] > 1:
            c["B"] //= 2
        else:
            c["n"] = max(10, c["n"] // 2)
    return c


def _frontiers(c):
    """Nodes expanded per drafted layer with the threshold off: the root, then min(n, k * the last)."""
    f = [1]
    for _ in range(min(c["D"], c["n"]) - 1):
        f.append(min(c["n"], f[-1] * c["k"]))
    return f


def _rows(c):
    """Draft rows of a whole pass that the path cannot do without."""
    if c["op"] == "rows":
        return c["rows"]
    if c["op"] == "pruned" or c["delta"] != "off":          # only what ends up in the tree is certain to be needed
        return c["B"] * (1 + c["n"])
    return c["B"] * sum(_frontiers(c))


def _logits(gen, rows, V, sigma, s):
    """Rows of draft logits: sigma * N(0, 1) and one peak per row, biased by a Zipf rank (the recipe of synth.draft_table)."""
    w = torch.arange(1, synth.ZIPF_TRUNC + 1, dtype=torch.float64, device="cuda") ** (-s)
    rank = torch.multinomial(w, rows, replacement=True, generator=gen).double() + 1.0
    bias = math.log(V) + 0.5 * sigma * sigma + synth.PEAK_B0 - torch.log(rank)
    peak = torch.randint(0, V, (rows,), device="cuda", generator=gen)
    out = torch.empty((rows, V), dtype=torch.bfloat16, device="cuda")
    for r0 in range(0, rows, 1024):
        r1 = min(rows, r0 + 1024)
        blk = torch.randn((r1 - r0, V), dtype=torch.float32, device="cuda", generator=gen).mul_(sigma)
        blk[torch.arange(r1 - r0, device="cuda"), peak[r0:r1]] += bias[r0:r1].float()
        out[r0:r1] = blk.bfloat16()
    return out


def _target(gen, draft, q):
    """The draft table with the argmax moved on a fraction q of the rows."""
    out = draft.clone()
    rows = torch.randperm(draft.shape[0], device="cuda", generator=gen)[: int(round(q * draft.shape[0]))]
    top = torch.stack([draft[r].argmax() for r in rows])
    other = torch.randint(0, draft.shape[1], (rows.numel(),), device="cuda", generator=gen)
    a, b = draft[rows, top], draft[rows, other]
    out[rows, top], out[rows, other] = b, a
    return out


def prepare(case, seed):
    c = dict(case)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    B, V, n, k, D = c["B"], c["V"], c["n"], c["k"], c["D"]
    i32 = dict(dtype=torch.int32, device="cuda")
    st = dict(op=c["op"], delta=OFF if c["delta"] == "off" else c["delta"], seed=seed)
    st["ot"] = ot = binding.OptTree(V, H, n, k, D, B)
    if c["op"] == "rows":
        st["draft"] = _logits(gen, H, V, c["sigma"], c["s"])
        st["rows"] = torch.randint(0, H, (c["rows"],), device="cuda", generator=gen).int()
        return st
    st["tree"] = ot.alloc_tree(B)
    if c["op"] == "layers":
        st["logits"] = [_logits(gen, B * f, V, c["sigma"], c["s"]).view(B, f, V) for f in _frontiers(c)]
        st["next"] = (torch.empty((B, n), **i32), torch.empty((B, n), **i32), torch.empty(B, **i32))
        return st
    st["draft"] = _logits(gen, H, V, c["sigma"], c["s"])
    st["target"] = _target(gen, st["draft"], c["q"])
    st["root"] = torch.randint(0, V, (B,), device="cuda", generator=gen).int()
    st["base"] = torch.randint(16, 2048, (B,), device="cuda", generator=gen).int()     # tokens before the step
    if c["op"] == "host":
        st["root"], st["base"] = st["root"].cpu().pin_memory(), st["base"].cpu().pin_memory()
        st["out"] = ot.alloc_host_out(B)
        return st
    st["mask"] = (torch.empty((B, n, ot.W), dtype=torch.int64, device="cuda"), torch.empty((B, n), **i32))
    st["accept"] = (torch.empty(B, **i32), torch.empty((B, D + 1), **i32), torch.empty((B, D), **i32), torch.empty(B, **i32))
    if c["op"] == "pruned":
        st["read"] = torch.empty(B, **i32)
        st["post"] = (torch.empty((B, n + 1, n + 1), dtype=torch.uint8, device="cuda"), torch.empty((B, D + 1), **i32),
                      torch.empty(B, **i32))
    return st


def _tree(t):
    return dict(token=t.token, parent=t.parent, depth=t.depth, phat=t.phat, n_sel=t.n_sel, depth_reached=t.depth_reached,
                expected_len=t.expected_len, esub_trace=t.esub_trace)


def run(st):
    ot, op, delta = st["ot"], st["op"], st["delta"]
    if op == "rows":
        return ot.row_softmax_topk(st["draft"], st["rows"])
    if op == "host":
        return ot.step_host(st["draft"], st["target"], st["root"], st["base"], delta, st["out"])
    tree = st["tree"]
    if op == "layers":
        ot.layers_begin(tree.token.shape[0])
        for x in st["logits"]:
            nxt = ot.layers_step(x, delta, tree, st["next"])
        return _tree(tree), nxt[2]                         # (a layer's tokens beyond its count are not written)
    if op == "pruned":
        ot.build_pruned(st["draft"], st["root"], delta, tree, st["read"])
    else:
        ot.build(st["draft"], st["root"], delta, tree)
    ot.mask(tree, st["base"], *st["mask"])
    if op == "sampled":
        ot.verify_sampled(tree, st["target"], st["root"], 1.0, st["seed"], 1, st["accept"])
    else:
        ot.verify(tree, st["target"], st["root"], st["accept"])
    out = [_tree(tree), st["mask"], st["accept"]]
    if op == "pruned":
        out += [st["read"], ot.post_verify(tree, st["mask"][0], st["accept"][0], st["accept"][2], st["post"])]
    return out


def work(case):
    """Every needed row of logits read once (the table stands in for a model: each expanded node has logits of its own), every
    output written once; about three operations per draft logit (scale, exponential, sum) and one comparison per target logit."""
    c = case
    B, V, n, D, W = c["B"], c["V"], c["n"], c["D"], (c["n"] + 63) // 64
    draft = _rows(c) * V
    if c["op"] == "rows":
        return dict(bytes=2 * draft + 4 * c["rows"] + 12 * c["rows"] * c["k"], flops=3 * draft)
    out = B * (n * 20 + 16 + 8 * D)
    if c["op"] == "layers":
        return dict(bytes=2 * draft + out + 4 * B, flops=3 * draft)
    target = B * (n + 1) * V
    out += B * (n * (8 * W + 4) + 8 + 4 * (2 * D + 1))
    if c["op"] == "pruned":
        out += B * ((n + 1) ** 2 + 4 * (D + 3))
    return dict(bytes=2 * (draft + target) + out + 8 * B, flops=3 * draft + target)


def tolerance(case):
    """Path values and E(A): products of up to max_depth probabilities whose softmax sums are formed in single precision.
    Against the same values in double precision the listed cases showed up to 3.8e-7 (2-norm) and 1.7e-6 (largest, depth 20);
    about four times that.  Whole numbers are decided by comparing path values, so a sequence may differ where two of them tie
    within rounding."""
    return dict(rel=1.5e-6, max=7e-6, differ=0.01)
