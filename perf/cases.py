"""What is measured: the calls that a user of this package makes, over the sizes that they are made at.

A case is a dict of plain values.  ``prepare`` makes what a program has in hand before the call,
``run`` makes the call through the package's public functions, ``work`` states what the call cannot
do without, ``tolerance`` how far another correct implementation may be off.

Kinds of call
    decode     one token for every sequence of a serving batch, fp32 state updated in place
    prefill    a prompt or a training sequence; dense or packed, with or without the block's value
               gate and feed-through, per-head gates or one set of gates for all heads
    backward   the gradients of a training step
    attention  sliding-window attention of the hybrid block
"""
import math

import numpy as np
import torch

import paper_2410_06577_b200 as rd


def _decode(name, n_seq, heads, dk=128, dv=256, block=False, shared=False):
    return {"name": name, "kind": "decode", "dtype": "bf16", "n_seq": n_seq, "heads": heads, "dk": dk, "dv": dv,
            "block": block, "shared": shared}


def _tokens(name, kind, batch, heads, length, dk=128, dv=256, dtype="bf16", lengths=None, gate_mean=-3.0,
            states=False, block=False, shared=False):
    """A dense batch of ``batch`` sequences of ``length`` tokens or, with ``lengths`` = (sequences, shortest,
    longest, seed of the lengths), sequences packed into one row of tokens."""
    n, lo, hi, seed = lengths or (0, 0, 0, 0)
    return {"name": name, "kind": kind, "dtype": dtype, "batch": batch, "heads": heads, "length": length, "dk": dk,
            "dv": dv, "packed": n, "shortest": lo, "longest": hi, "lengths_seed": seed, "gate_mean": gate_mean,
            "states": states, "block": block, "shared": shared}


def _attention(name, batch, heads, length, window):
    return {"name": name, "kind": "attention", "dtype": "bf16", "batch": batch, "heads": heads, "length": length,
            "window": window, "d": 128}


def listed():
    return [
        # One user's next token in one layer: nothing but latency, the launch and the host's part of the call.
        _decode("decode_one", 1, 16),
        # A serving batch's next token (the benchmark's decode workload): a stream of fp32 states.
        _decode("decode_batch", 256, 16),
        # The smallest prefill, in fp32, the data type for checking a model (the benchmark's smallest workload).
        _tokens("prefill_f32", "prefill", 1, 1, 256, dk=64, dv=64, dtype="f32"),
        # A prompt of odd length in the whole block (value gate and feed-through): a single user waits for it.
        _tokens("prefill_prompt", "prefill", 1, 16, 777, block=True),
        # A layer's forward pass over a training batch (the benchmark's headline workload).
        _tokens("prefill_layer", "prefill", 4, 16, 2048),
        # A long document continued from a state: one sequence, long memory, few heads for the device.
        _tokens("prefill_long", "prefill", 1, 16, 32768, gate_mean=-4.0, states=True),
        # A batch of requests or documents of very different lengths packed together.
        _tokens("prefill_packed", "prefill", 1, 16, 0, lengths=(64, 128, 4096, 4)),
        # The layout that the paper writes the block in: 64 key channels, one set of gates for all value columns.
        _tokens("prefill_paper_layout", "prefill", 4, 16, 2048, dk=64, shared=True),
        # A layer's backward pass over the training batch.
        _tokens("backward_layer", "backward", 4, 16, 2048),
        # The backward pass over a few packed documents, with gradients of the final and initial states.
        _tokens("backward_packed", "backward", 1, 16, 0, lengths=(7, 50, 600, 7), states=True),
        # The hybrid block's attention over a training batch, window of half the context.
        _attention("attention_layer", 4, 16, 2048, 1024),
        # The same for one long prompt of odd length.
        _attention("attention_prompt", 1, 16, 5001, 2048),
    ]


def _spread(rng, lo, hi):
    """A whole number of lo..hi, even over the logarithm; odd ones come up as often as even ones."""
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 0.49)))))))


def draw(rng):
    kind = rng.choice(["decode", "prefill", "prefill", "prefill_packed", "backward", "attention"])
    heads = rng.choice([4, 8, 16, 16, 32])
    if kind == "decode":
        dk, dv = rng.choice([(128, 256), (128, 256), (64, 256), (128, 128)])
        return _decode("", _spread(rng, 1, 4096 // heads), heads, dk, dv, block=rng.random() < 0.3,
                       shared=rng.random() < 0.3)
    if kind == "prefill":
        if rng.random() < 0.15:                                           # fp32: small, for checking
            return _tokens("", kind, _spread(rng, 1, 3), rng.randint(1, 4), _spread(rng, 16, 1024), dk=64,
                           dv=rng.choice([64, 128]), dtype="f32", states=rng.random() < 0.5)
        dk, dv, shared = rng.choice([(128, 256, False), (128, 256, False), (128, 512, False), (128, 128, False),
                                     (128, 256, True), (64, 256, True)])
        most = 131072 if dk == 64 else 524288                             # (token, head) pairs of 256 value columns
        length = _spread(rng, 32, min(32768, most * 256 // (heads * dv)))
        batch = _spread(rng, 1, max(1, min(16, most * 256 // (heads * dv * length))))
        block = dv != 128 and dk == 128 and rng.random() < 0.3
        return _tokens("", kind, batch, heads, length, dk=dk, dv=dv, gate_mean=rng.choice([-3.0, -4.0]),
                       states=rng.random() < 0.4, block=block, shared=shared)
    if kind == "prefill_packed":
        longest = _spread(rng, 128, 4096)
        n = _spread(rng, 2, max(2, min(256, 2 * 1048576 // (heads * longest))))
        return _tokens("", "prefill", 1, heads, 0, lengths=(n, _spread(rng, 1, 128), longest, rng.randint(0, 10 ** 6)),
                       states=rng.random() < 0.4)
    if kind == "backward":
        if rng.random() < 0.4:
            longest = _spread(rng, 128, 2048)
            n = _spread(rng, 2, max(2, min(64, 2 * 131072 // (heads * longest))))
            return _tokens("", kind, 1, heads, 0, lengths=(n, _spread(rng, 1, 128), longest, rng.randint(0, 10 ** 6)),
                           states=rng.random() < 0.4)
        length = _spread(rng, 64, min(4096, 131072 // heads))
        batch = _spread(rng, 1, max(1, min(8, 131072 // (heads * length))))
        return _tokens("", kind, batch, heads, length, states=rng.random() < 0.4)
    length = _spread(rng, 64, 8192)
    batch = _spread(rng, 1, max(1, min(8, 131072 // (heads * length))))
    return _attention("", batch, heads, length, _spread(rng, 64, 4096))


def _lengths(case):
    """Lengths of the sequences of a prefill or backward case."""
    if not case["packed"]:
        return [case["length"]] * case["batch"]
    rng = np.random.default_rng(case["lengths_seed"])
    return [int(n) for n in rng.integers(case["shortest"], case["longest"] + 1, case["packed"])]


class _Maker:
    """Seeded normal values on the GPU, in the dtype of the tokens unless said otherwise."""

    def __init__(self, seed, dtype):
        self.gen = torch.Generator(device="cuda")
        self.gen.manual_seed(seed)
        self.dtype = torch.bfloat16 if dtype == "bf16" else torch.float32

    def normal(self, *shape, mean=0.0, std=1.0, dtype=None):
        t = torch.randn(shape, generator=self.gen, device="cuda", dtype=torch.float32)
        if std != 1.0:
            t.mul_(std)
        if mean != 0.0:
            t.add_(mean)
        return t.to(dtype or self.dtype)

    def gate(self, *shape):
        """The value gate after its sigmoid, in (0, 1)."""
        return torch.sigmoid(self.normal(*shape, dtype=torch.float32)).to(self.dtype)


def prepare(case, seed):
    m = _Maker(seed, case["dtype"])
    st = {"kind": case["kind"]}
    if case["kind"] == "attention":
        b, h, t, d = case["batch"], case["heads"], case["length"], case["d"]
        st.update(q=m.normal(b, h, t, d), k=m.normal(b, t, d), v=m.normal(b, h, t, d), window=case["window"])
        return st
    h, dk, dv = case["heads"], case["dk"], case["dv"]
    hq = 1 if case["shared"] else h
    std = dk ** -0.5
    if case["kind"] == "decode":
        lead, lead_q, tail = (case["n_seq"], h), (case["n_seq"], hq), ()
        gate_mean, n_seq = -3.0, case["n_seq"]
        st["state"] = m.normal(n_seq, h, dk, dv, std=0.1, dtype=torch.float32)
    else:
        lengths = _lengths(case)
        b, t = (1, sum(lengths)) if case["packed"] else (case["batch"], case["length"])
        lead, lead_q, tail = (b, h), (b, hq), (t,)
        gate_mean, n_seq = case["gate_mean"], len(lengths)
        st["cu_seqlens"] = None
        if case["packed"]:
            st["cu_seqlens"] = torch.tensor(np.concatenate([[0], np.cumsum(lengths)]), dtype=torch.int32, device="cuda")
        st["s0"] = m.normal(n_seq, h, dk, dv, std=0.1, dtype=torch.float32) if case["states"] else None
    st["tokens"] = (m.normal(*lead_q, *tail, dk, std=std), m.normal(*lead_q, *tail, dk, std=std),
                    m.normal(*lead_q, *tail, dk, mean=gate_mean), m.normal(*lead_q, *tail, dk),
                    m.normal(*lead, *tail, dv))                           # q, k, x, y, v
    st["block"] = {}
    if case["block"]:
        st["block"] = {"beta_hat": m.gate(*lead, *tail, dv), "feed_d": m.normal(h, dv, dtype=torch.float32),
                       "feed_x": m.normal(*lead, *tail, dv)}
    if case["kind"] == "backward":
        st["d_o"] = m.normal(*lead, *tail, dv)
        st["states"] = case["states"]
        st["d_sT"] = m.normal(n_seq, h, dk, dv, std=0.1, dtype=torch.float32) if case["states"] else None
    return st


def run(state):
    kind = state["kind"]
    if kind == "attention":
        return rd.swska_fwd(state["q"], state["k"], state["v"], state["window"])
    q, k, x, y, v = state["tokens"]
    if kind == "decode":
        o = rd.ddts_step(q, k, x, y, v, state["state"], **state["block"])
        return o, state["state"]
    if kind == "prefill":
        return rd.ddts_fwd(q, k, x, y, v, state["s0"], cu_seqlens=state["cu_seqlens"], **state["block"])
    g = rd.ddts_bwd(q, k, x, y, v, state["d_o"], state["s0"], state["d_sT"], cu_seqlens=state["cu_seqlens"],
                    want_d_s0=state["states"])
    return {name: t for name, t in g.items() if t is not None}


def work(case):
    """Each input read once and each output written once; the arithmetic of the recurrence as it is stated
    (two multiply-adds per state element and token forwards, five backwards), of the attention's visible pairs."""
    size = 2 if case["dtype"] == "bf16" else 4
    if case["kind"] == "attention":
        b, h, t, w, d = case["batch"], case["heads"], case["length"], case["window"], case["d"]
        pairs = t * (t + 1) // 2 if t <= w else w * (w + 1) // 2 + (t - w) * w
        return {"bytes": size * d * b * t * (3 * h + 1), "flops": 4 * d * pairs * b * h}
    h, dk, dv = case["heads"], case["dk"], case["dv"]
    hq = 1 if case["shared"] else h
    if case["kind"] == "decode":
        tokens, states = case["n_seq"], 2 * case["n_seq"]
    else:
        lengths = _lengths(case)
        tokens, states = sum(lengths), len(lengths) * (2 if case["states"] else 1)
    per_key, per_value, updates = 4, 2, 2                     # q, k, x, y; v, o
    if case["block"]:
        per_value += 2
    if case["kind"] == "backward":
        per_key, per_value, updates = 8, 3, 5                 # and their gradients; v, d_o, d_v
        states = len(lengths) * (3 if case["states"] else 0)
    return {"bytes": size * tokens * (per_key * hq * dk + per_value * h * dv) + 4 * states * h * dk * dv,
            "flops": 2 * updates * tokens * h * dk * dv}


# Relative error against a 64-bit computation of the same equations, as measured at these sizes (the
# worst output of each kind), times four.  bf16 results alone carry 1.7e-3 of rounding.
_BF16_REL = {"decode": 7e-3,       # 1.7e-3: the rounding of the output
             "prefill": 1.3e-2,    # 3.3e-3: operands of the contractions and the output in bf16
             "backward": 8e-3,     # 1.9e-3
             "attention": 9e-3}    # 2.1e-3: probabilities and the output in bf16


def tolerance(case):
    if case["dtype"] == "f32":
        return {"rel": 1e-5}       # 2.4e-7 measured; sums of up to 64 + 64 products in any order
    return {"rel": _BF16_REL[case["kind"]]}
