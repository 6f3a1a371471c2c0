"""The work that users of the library time: the quantised linear layers of one model block, call by call.

A case is one pass of a serving or prefill program over
  "linear"  one weight matrix through uniql_qlinear, fp16;
  "layer"   the linears of one transformer decoder layer: q|k|v projection with the pruned rotary embedding, output
            projection on the kept channels of every head, SwiGLU MLP block (three calls);
  "mamba"   the linears of one Mamba2 mixer: in_proj with z and x rows pruned per SSM head, out_proj on the kept
            channels of every head (two calls);
  "head"    both ends of a language model: 4-bit embedding rows, lm_head over the whole vocabulary (two calls).
Attention, scan and normalisation are not part of the library: what they would hand over is made by prepare().

"rows" is the number of tokens of the pass (1: one sequence being decoded, 4 .. 128: a batch of sequences being
decoded, above: prompts), "keep" the share of channels that the pruning rate chosen at run time leaves.
"""
import math

import torch

from paper_2512_03383_b200 import binding as B
from paper_2512_03383_b200 import synth

GROUP = 128
DTYPES = {"f16": torch.float16, "bf16": torch.bfloat16}

#: Transformer shapes; Qwen2.5's q, k and v projections carry biases, Llama-3's do not.
LAYERS = {
    "llama3-8b": dict(s=synth.LLAMA3_8B, bias=False),
    "qwen2.5-7b": dict(s=synth.QWEN25_7B, bias=True),
}
#: Mamba2 mixers: Mamba2-2.7B, and the one of a hybrid model's layer (Bamba-v2-9B).
MIXERS = {
    "mamba2-2.7b": dict(hidden=2560, d_inner=5120, nheads=80),
    "bamba-v2-9b": dict(hidden=4096, d_inner=8192, nheads=128),
}
HEADDIM, D_STATE = 64, 128
VOCAB, VOCAB_HIDDEN = 128256, 4096


def listed():
    return [
        # the smallest call: one matrix, one token (what a single launch costs its caller)
        {"name": "linear-1", "op": "linear", "n": 2048, "k": 2048, "rows": 1, "keep": 0.85},
        # a chat with one user, un-pruned: one generated token
        {"name": "llama-1", "op": "layer", "model": "llama3-8b", "rows": 1, "keep": 1.0, "dtype": "f16"},
        # a few users at once (or a few drafted tokens to verify), the strongest pruning rate of the paper's tables
        {"name": "llama-4-pruned", "op": "layer", "model": "llama3-8b", "rows": 4, "keep": 0.65, "dtype": "f16"},
        # the same for a model that is kept in bf16, as it was published
        {"name": "qwen-2-bf16", "op": "layer", "model": "qwen2.5-7b", "rows": 2, "keep": 0.85, "dtype": "bf16"},
        # a small serving batch
        {"name": "llama-16", "op": "layer", "model": "llama3-8b", "rows": 16, "keep": 0.75, "dtype": "f16"},
        # one generated token of a state-space model
        {"name": "mamba-1", "op": "mamba", "model": "mamba2-2.7b", "rows": 1, "keep": 0.85, "dtype": "f16"},
        # first and last matrix of a decoding step of eight sequences
        {"name": "head-8", "op": "head", "rows": 8, "dtype": "f16"},
        # a large serving batch: the range between decoding one sequence and reading prompts
        {"name": "llama-64", "op": "layer", "model": "llama3-8b", "rows": 64, "keep": 0.85, "dtype": "f16"},
        # a short prompt
        {"name": "llama-512", "op": "layer", "model": "llama3-8b", "rows": 512, "keep": 0.75, "dtype": "f16"},
        # prompts of a state-space model
        {"name": "mamba-1024", "op": "mamba", "model": "mamba2-2.7b", "rows": 1024, "keep": 0.75, "dtype": "f16"},
        # a prompt of no particular length in bf16
        {"name": "qwen-677-bf16", "op": "layer", "model": "qwen2.5-7b", "rows": 677, "keep": 0.65, "dtype": "bf16"},
        # the largest: a long prompt, un-pruned
        {"name": "qwen-2048-bf16", "op": "layer", "model": "qwen2.5-7b", "rows": 2048, "keep": 1.0, "dtype": "bf16"},
    ]


def draw(rng):
    op = rng.choices(["layer", "mamba", "linear", "head"], [5, 2, 2, 1])[0]
    rows = _log_int(rng, 1, 2048)
    keep = rng.choice([1.0, 0.85, 0.75, 0.65, round(rng.uniform(0.55, 1.0), 3)])
    if op == "linear":
        return {"op": op, "n": 8 * _log_int(rng, 64, 1792), "k": GROUP * _log_int(rng, 8, 112), "rows": rows, "keep": keep}
    if op == "head":
        return {"op": op, "rows": min(rows, _log_int(rng, 1, 128)), "dtype": rng.choice(["f16", "bf16"])}
    model = rng.choice(sorted(LAYERS if op == "layer" else MIXERS))
    return {"op": op, "model": model, "rows": rows, "keep": keep, "dtype": rng.choice(["f16", "bf16"])}


def _log_int(rng, lo, hi):
    return min(hi, max(lo, round(math.exp(rng.uniform(math.log(lo), math.log(hi + 1))))))


# ----------------------------------------------------------------------------- sizes
def _keep8(rate, dim):
    """Kept channels of a long dimension: the nearest multiple of 8 (the SwiGLU block asks for that at decode sizes)."""
    return min(dim, 8 * round(rate * dim / 8))


def _matrices(case):
    """(stored rows, stored columns, kept rows, kept columns) of every weight matrix of the pass, in its order."""
    op, keep = case["op"], case.get("keep", 1.0)
    if op == "linear":
        return [(case["n"], case["k"], _keep8(keep, case["n"]), _keep8(keep, case["k"]))]
    if op == "head":
        return [(VOCAB, VOCAB_HIDDEN, VOCAB, VOCAB_HIDDEN)]
    if op == "mamba":
        m = MIXERS[case["model"]]
        hd = synth.keep_count(keep, HEADDIM)
        rest = 2 * D_STATE + m["nheads"]
        return [(2 * m["d_inner"] + rest, m["hidden"], 2 * m["nheads"] * hd + rest, m["hidden"]),
                (m["hidden"], m["d_inner"], m["hidden"], m["nheads"] * hd)]
    s = LAYERS[case["model"]]["s"]
    hd, inter = synth.keep_count(keep, s.head_dim), _keep8(keep, s.intermediate)
    q, kv = s.n_q_heads, s.n_kv_heads
    return [(q * s.head_dim, s.hidden, q * hd, s.hidden), (kv * s.head_dim, s.hidden, kv * hd, s.hidden),
            (kv * s.head_dim, s.hidden, kv * hd, s.hidden), (s.hidden, q * s.head_dim, s.hidden, q * hd),
            (s.intermediate, s.hidden, inter, s.hidden), (s.intermediate, s.hidden, inter, s.hidden),
            (s.hidden, s.intermediate, s.hidden, inter)]


def work(case):
    """Kept weights once (4-bit codes, an fp16 scale and zero-point per 128), inputs and outputs once."""
    rows, total_b, total_f = case["rows"], 0.0, 0.0
    for _, _, n, k in _matrices(case):
        total_b += n * k * (0.5 + 4 / GROUP)
        total_f += 2.0 * rows * n * k
    if case["op"] == "linear":
        _, _, n, k = _matrices(case)[0]
        columns = n + k
    elif case["op"] == "head":       # embedding rows (codes, scales and zero-points; out), hidden states, logits
        total_b += rows * VOCAB_HIDDEN * (0.5 + 4 / GROUP)
        columns = VOCAB_HIDDEN + VOCAB_HIDDEN + VOCAB
    elif case["op"] == "mamba":
        (_, _, n1, k1), (_, _, n2, k2) = _matrices(case)
        columns = n1 + k1 + n2 + k2
    else:
        (_, _, q, hidden), (_, _, kv, _), _, (_, _, _, ctx), (_, _, inter, _), _, _ = _matrices(case)
        columns = hidden + q + 2 * kv + ctx + hidden + hidden + inter + hidden    # x, q, k, v, ctx, o, x, h, y
    return {"bytes": total_b + 2.0 * rows * columns, "flops": total_f}


def tolerance(case):
    """fp32 sums of 4-bit weights times 16-bit activations, rounded once to the output type (twice along the SwiGLU
    block, whose h is a stored tensor): two correct implementations differ by that rounding, and in fp16 by the rounding
    of an fp16 or a 16-bit fixed-point operand beside it."""
    if case.get("dtype", "f16") == "bf16":
        return {"rel": 5e-3, "max": 4e-2}
    return {"rel": 1e-3, "max": 1e-2}


# ----------------------------------------------------------------------------- inputs
class _Draw:
    """Everything random of a state, from one seed, made on the GPU."""

    def __init__(self, seed, dtype):
        self.g = torch.Generator(device="cuda").manual_seed(seed)
        self.dtype = dtype

    def weight(self, n, k, std=0.02):
        """N(0, std) quantised to asymmetric uint4 per 128 input channels, low nibble first."""
        packed = torch.empty((n, k // 2), dtype=torch.uint8, device="cuda")
        scales = torch.empty((n, k // GROUP), dtype=torch.float16, device="cuda")
        zeros = torch.empty_like(scales)
        step = max(1, (64 << 20) // k)
        for r in range(0, n, step):
            w = torch.randn((min(step, n - r), k // GROUP, GROUP), generator=self.g, device="cuda") * std
            lo, hi = torch.aminmax(w, dim=2, keepdim=True)
            s = ((hi - lo) / 15).half()
            z = torch.round(-lo / s.float()).clamp_(0, 15)
            c = (torch.round(w / s.float()) + z).clamp_(0, 15).to(torch.uint8).view(-1, k)
            packed[r:r + step] = c[:, 0::2] | (c[:, 1::2] << 4)
            scales[r:r + step] = s.view(-1, k // GROUP)
            zeros[r:r + step] = z.view(-1, k // GROUP).half()
        return packed, scales, zeros

    def x(self, rows, k):
        """Activations ~N(0, 1) with one channel of a hundred scaled by 20, as LLM hidden states have."""
        x = torch.randn((rows, k), generator=self.g, device="cuda")
        loud = torch.rand(k, generator=self.g, device="cuda").argsort()[:max(1, k // 100)]
        x[:, loud] *= 20
        return x.to(self.dtype)

    def bias(self, n):
        return (torch.randn(n, generator=self.g, device="cuda") * 0.5).to(self.dtype)

    def ints(self, hi, *shape):
        return torch.randint(0, hi, shape, generator=self.g, device="cuda", dtype=torch.int32)

    def kept_pairs(self, heads, half, keep):
        """Original indices of the rotation pairs that every key-value head keeps."""
        return torch.rand((heads, half), generator=self.g, device="cuda").argsort(dim=1)[:, :keep].int().contiguous()

    def out(self, rows, n):
        return torch.zeros((rows, n), dtype=self.dtype, device="cuda")


def prepare(case, seed):
    rows, op = case["rows"], case["op"]
    d = _Draw(seed, DTYPES[case.get("dtype", "f16")])
    st = {"op": op, "rows": rows, "w": [d.weight(n, k) for n, k, _, _ in _matrices(case)], "sizes": _matrices(case)}
    if op == "linear":
        n, k = st["sizes"][0][2:]
        st.update(x=d.x(rows, k), y=d.out(rows, n))
    elif op == "head":
        st.update(table=d.weight(VOCAB, VOCAB_HIDDEN), ids=d.ints(VOCAB, rows), e=d.out(rows, VOCAB_HIDDEN),
                  x=d.x(rows, VOCAB_HIDDEN), y=d.out(rows, VOCAB))
    elif op == "mamba":
        m = MIXERS[case["model"]]
        hd = synth.keep_count(case["keep"], HEADDIM)
        (_, _, n1, k1), (_, _, n2, k2) = st["sizes"]
        st.update(x=d.x(rows, k1), zxbcdt=d.out(rows, n1), scanned=d.x(rows, k2), y=d.out(rows, n2),
                  in_rows=synth.map_mamba_in_proj(m["d_inner"], HEADDIM, hd, D_STATE, 1, m["nheads"]),
                  out_cols=synth.map_per_head(m["nheads"], HEADDIM, hd))
    else:
        s, bias = LAYERS[case["model"]]["s"], LAYERS[case["model"]]["bias"]
        hd = synth.keep_count(case["keep"], s.head_dim)
        inter = st["sizes"][4][2]
        pitch = (inter + 63) // 64 * 64      # whole 128-byte lines, as the header advises
        q, kv = s.n_q_heads * hd, s.n_kv_heads * hd
        st.update(s=s, hd=hd, inter=inter, pitch=pitch, pos=d.ints(8192, rows),
                  idx=d.kept_pairs(s.n_kv_heads, s.head_dim // 2, hd // 2),
                  bias=[d.bias(st["sizes"][j][0]) if bias else None for j in range(3)],
                  x=d.x(rows, s.hidden), q=d.out(rows, q), k=d.out(rows, kv), v=d.out(rows, kv),
                  ctx=d.x(rows, q), ctx_cols=synth.map_per_head(s.n_q_heads, s.head_dim, hd), o=d.out(rows, s.hidden),
                  x2=d.x(rows, s.hidden), h=d.out(rows, pitch)[:, :inter], y=d.out(rows, s.hidden))
    return st


# ----------------------------------------------------------------------------- one pass
def run(st):
    return {"linear": _linear, "head": _head, "mamba": _mamba, "layer": _layer}[st["op"]](st)


def _linear(st):
    n, k, n_kept, k_kept = st["sizes"][0]
    B.qlinear(st["x"], *st["w"][0], st["rows"], k, n, k_kept, n_kept, st["y"])
    return st["y"]


def _head(st):
    B.embed_rows(*st["table"], st["ids"], st["e"])
    B.qlinear_ex(st["x"], VOCAB_HIDDEN, *st["w"][0], None, st["rows"], VOCAB_HIDDEN, VOCAB, None, VOCAB_HIDDEN, None,
                 VOCAB, st["y"], VOCAB)
    return st["e"], st["y"]


def _mamba(st):
    (n1, k1, n1_kept, _), (n2, k2, _, k2_kept) = st["sizes"]
    B.qlinear_ex(st["x"], k1, *st["w"][0], None, st["rows"], k1, n1, None, k1, st["in_rows"], 0, st["zxbcdt"], n1_kept)
    B.qlinear_ex(st["scanned"], k2_kept, *st["w"][1], None, st["rows"], k2, n2, st["out_cols"], 0, None, n2, st["y"], n2)
    return st["zxbcdt"], st["y"]


def _layer(st):
    s, hd, rows, w = st["s"], st["hd"], st["rows"], st["w"]
    q, kv = s.n_q_heads * hd, s.n_kv_heads * hd
    B.qkv_rope_proj(st["x"], s.hidden, *w[0], *w[1], *w[2], *st["bias"], rows, s.hidden, s.n_q_heads, s.n_kv_heads,
                    s.head_dim, hd, hd, st["idx"], st["pos"], s.theta, None, st["q"], q, st["k"], kv, st["v"], kv)
    B.qlinear_ex(st["ctx"], q, *w[3], None, rows, s.n_q_heads * s.head_dim, s.hidden, st["ctx_cols"], 0, None, s.hidden,
                 st["o"], s.hidden)
    B.mlp_swiglu(st["x2"], s.hidden, *w[4], *w[5], *w[6], rows, s.hidden, s.intermediate, st["inter"], st["h"],
                 st["pitch"], st["y"], s.hidden)
    return st["q"], st["k"], st["v"], st["o"], st["h"], st["y"]
