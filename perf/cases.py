"""The work that users of the library have it do, as measurable cases.

A case is one call pattern of a program that holds an E2-TTT layer, through the public binding:

  decode    e2ttt_apply: the outputs of fixed fast weights for the next tokens of every sequence
  forward   e2ttt_chunk_fwd (or its post-chunk-normalised form): a prefill, or the update of one accumulated chunk
  train     the forward with saved states (or checkpoints of them) and the reverse pass on them: one layer's training step
  prepare   e2ttt_prepare_fwd and e2ttt_prepare_bwd: q / k normalisation and gates from their logits, and the adjoints

Shapes are those of the benchmark configurations and tests: head dimension 64 or 128 with a hidden width of 4 d (GELU-MLP) or
8 d / 3 rounded up to a multiple of 64 (SwiGLU), chunks of 16 to 512 tokens (the method trains with 512, the layer benchmark
runs 64), 1 to 16 heads and a batch of 1 to 8, sequences of one token to 8192; other widths, chunk sizes and ragged
lengths are what the any-shape promise of the interface stands for.  bf16 I/O is what models run in; fp32 I/O is the
checking mode and is used on small problems.

Values: q and k are SiLU + L2-normalised rows (what the preparation step hands over), v and output gradients are N(0, 1), fast
weights N(0, 0.02), gates in the regime models train in (learning rate up to 0.01, momentum sigmoid^(1/32), decay strength up to 0.1).
"""
from __future__ import annotations

import math

import torch

from paper_2608_21308_b200 import binding as E
from paper_2608_21308_b200.inputs import mat_shapes, swiglu_hidden

GATES = (0.01, 32.0, 0.1, 1e-12)  # eta_base, tau, alpha_base, norm_eps
LN_EPS = 1e-5
NORM_EPS = 1e-5


def _case(name, op, kind, B, H, L, d, h, C, io="bf16", ckpt=0, normed=False):
    c = {"op": op, "kind": kind, "B": B, "H": H, "L": L, "d": d, "h": h, "C": C, "io": io, "ckpt": ckpt, "normed": normed}
    return dict(c, name=name) if name else c


def listed():
    return [
        # one token for each of 16 heads of one request: the smallest call there is, launch and host latency
        _case("decode batch 1", "decode", "mlp", 1, 16, 1, 128, 512, 1),
        # the same for eight requests, SwiGLU fast weights: reads 75 MB of state
        _case("decode batch 8 swiglu", "decode", "swiglu", 8, 16, 1, 128, 384, 1),
        # what a decoder does every 64 tokens: the chunk update of the tokens that accumulated, with a momentum state
        _case("decode chunk update", "forward", "mlp", 4, 16, 64, 128, 512, 64),
        # prefill at the 1.3B layer shape
        _case("prefill 1.3B", "forward", "mlp", 4, 16, 4096, 128, 512, 64),
        # prefill of a ragged prompt, SwiGLU fast weights
        _case("prefill swiglu ragged", "forward", "swiglu", 4, 16, 1000, 128, 384, 64),
        # prefill at the 125M layer shape
        _case("prefill 125M", "forward", "mlp", 8, 12, 2048, 64, 256, 64),
        # prefill with the chunk size the method is trained with
        _case("prefill chunk 512", "forward", "mlp", 4, 16, 4096, 128, 512, 512),
        # training step at the 1.3B layer shape
        _case("train 1.3B", "train", "mlp", 4, 16, 4096, 128, 512, 64),
        # training step as the method trains: 2K tokens, chunks of 512, post-chunk normalisation, SwiGLU
        _case("train chunk 512 swiglu normed", "train", "swiglu", 2, 16, 2048, 128, 384, 512, normed=True),
        # long-context training step: one long sequence, 16 heads, state checkpoints every 32 chunks
        _case("train long context", "train", "mlp", 1, 16, 8192, 128, 512, 64, ckpt=32),
        # the fp32 checking mode, forward and reverse pass of the tiny configuration
        _case("check fp32", "train", "mlp", 1, 1, 256, 64, 256, 16, io="f32"),
        # token preparation and its reverse pass over the tokens of the 1.3B layer shape
        _case("prepare tokens", "prepare", "mlp", 4, 16, 4096, 128, 512, 64),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _hidden(kind, d):
    return 4 * d if kind == "mlp" else swiglu_hidden(d)


def draw(rng):
    op = rng.choice(["decode", "forward", "forward", "train", "train", "prepare"])
    kind = rng.choice(["mlp", "mlp", "swiglu"])
    # widths: mostly the two model shapes; sometimes another head dimension or hidden width
    d = rng.choice([64, 128, 128, 128, rng.choice([48, 72, 80, 96, 112])])
    h = _hidden(kind, d)
    if rng.random() < 0.2:
        h = 8 * rng.randint(8, 64)
    B, H = _log_int(rng, 1, 8), _log_int(rng, 2, 16)
    if op == "decode":
        return _case(None, op, kind, B, H, rng.choice([1, 1, 1, 2, 5]), d, h, 1, io=rng.choice(["bf16", "bf16", "bf16", "f32"]))
    if op == "prepare":
        return _case(None, op, kind, B, H, _log_int(rng, 64, 4096), d, h, 64, io=rng.choice(["bf16", "bf16", "bf16", "f32"]))
    if rng.random() < 0.15:  # fp32 checking mode: small problems
        C = rng.choice([16, 24, 32, 64])
        return _case(None, op, kind, 1, rng.randint(1, 4), C * rng.randint(1, 8) + rng.choice([0, 0, 7]), rng.choice([48, 64, 64, 72]),
                     rng.choice([128, 192, 200, 256]), C, io="f32")
    C = rng.choice([16, 32, 64, 64, 64, 128, 256, 512, 512, rng.choice([24, 40, 96, 200])])
    # SwiGLU states amplify rounding from chunk to chunk: sequences short enough that results stay comparable
    L = min(C * _log_int(rng, 1, 64 if kind == "mlp" else 12), 4096)
    if rng.random() < 0.4:
        L = max(1, L - rng.randint(1, C - 1))
    normed = rng.random() < 0.2
    ckpt = rng.choice([0, 0, 4, 8]) if op == "train" and not normed else 0
    return _case(None, op, kind, min(B, 4), H, L, d, h, C, ckpt=ckpt, normed=normed)


def _kind(case):
    return E.E2TTT_MLP_GELU if case["kind"] == "mlp" else E.E2TTT_SWIGLU


def prepare(case, seed):
    B, H, L, d, h, C = (case[n] for n in ("B", "H", "L", "d", "h", "C"))
    kind, dev = _kind(case), "cuda"
    io = torch.float32 if case["io"] == "f32" else torch.bfloat16
    g = torch.Generator(device=dev)
    g.manual_seed(seed)

    def randn(*shape):
        return torch.randn(shape, generator=g, device=dev, dtype=torch.float32)

    p = E.make_params(B, H, L, d, h, C, kind, E.E2TTT_F32 if case["io"] == "f32" else E.E2TTT_BF16, LN_EPS, E.E2TTT_IMPL_AUTO,
                      case["ckpt"])
    gp = E.e2ttt_gate_params(*GATES)
    s = {"op": case["op"], "normed": case["normed"], "p": p, "gp": gp}
    if case["op"] == "decode":
        s["q"] = torch.nn.functional.normalize(torch.nn.functional.silu(randn(B, H, L, d)), dim=-1).to(io)
        s["W"] = [0.02 * randn(B, H, r, c) for r, c in mat_shapes(kind, d, h)]
        s["o"] = torch.empty_like(s["q"])
        return s
    if case["op"] == "prepare":
        s["q_raw"], s["k_raw"] = randn(B, H, L, d).to(io), randn(B, H, L, d).to(io)
        s["logits"] = [randn(B, H, L), 1.0 + randn(B, H, L), 3.0 + randn(B, H, L)]
        s["q"], s["k"] = torch.empty_like(s["q_raw"]), torch.empty_like(s["q_raw"])
        s["gates"] = [torch.empty_like(x) for x in s["logits"]]
        s["dq"], s["dk"] = randn(B, H, L, d).to(io), randn(B, H, L, d).to(io)
        s["d_gates"] = [randn(B, H, L) for _ in range(3)]
        s["d_raw"] = [torch.empty_like(s["q_raw"]) for _ in range(2)]
        s["d_logits"] = [torch.empty_like(x) for x in s["logits"]]
        return s
    train = case["op"] == "train"
    s["q"], s["k"] = (torch.nn.functional.normalize(torch.nn.functional.silu(randn(B, H, L, d)), dim=-1).to(io) for _ in range(2))
    s["v"] = randn(B, H, L, d).to(io)
    eta = GATES[0] * torch.sigmoid(randn(B, H, L))
    beta = torch.sigmoid(1.0 + randn(B, H, L)) ** (1.0 / GATES[1])
    s["gates"] = [eta, beta, 1.0 - eta * GATES[2] * torch.sigmoid(3.0 + randn(B, H, L))]
    shapes = mat_shapes(kind, d, h)
    s["W"] = [0.02 * randn(B, H, r, c) for r, c in shapes]
    # a sequence starts without momentum; the update of one chunk in the middle of a sequence has one
    s["M"] = [0.002 * randn(B, H, r, c) for r, c in shapes] if not train and L <= C else None
    s["norm"] = [w.norm(dim=-1).contiguous() for w in s["W"]] if case["normed"] else None
    s["o"] = torch.empty_like(s["q"])
    s["Wf"], s["Mf"] = [torch.empty_like(w) for w in s["W"]], [torch.empty_like(w) for w in s["W"]]
    size = E.e2ttt_workspace_bytes_normed if case["normed"] else E.e2ttt_workspace_bytes
    s["ws"] = torch.empty(size(p, int(train)), dtype=torch.uint8, device=dev)
    if train:
        s["d_o"] = randn(B, H, L, d).to(io)
        s["d_qkv"] = [torch.empty_like(s["q"]) for _ in range(3)]
        s["d_gates"] = [torch.empty_like(eta) for _ in range(3)]
        s["dW"], s["dM"] = [torch.empty_like(w) for w in s["W"]], [torch.empty_like(w) for w in s["W"]]
        s["d_norm"] = [torch.empty_like(n) for n in s["norm"]] if case["normed"] else None
    return s


def run(s):
    p, op = s["p"], s["op"]
    if op == "decode":
        E.e2ttt_apply(p, s["q"], s["W"], s["o"])
        return s["o"]
    if op == "prepare":
        E.e2ttt_prepare_fwd(p, s["gp"], s["q_raw"], s["k_raw"], *s["logits"], s["q"], s["k"], *s["gates"])
        E.e2ttt_prepare_bwd(p, s["gp"], s["q_raw"], s["k_raw"], *s["logits"], s["dq"], s["dk"], *s["d_gates"], *s["d_raw"],
                            *s["d_logits"])
        return {"q": s["q"], "k": s["k"], "gates": s["gates"], "d_raw": s["d_raw"], "d_logits": s["d_logits"]}
    train = op == "train"
    if s["normed"]:
        E.e2ttt_chunk_fwd_normed(p, s["q"], s["k"], s["v"], *s["gates"], s["W"], s["M"], s["norm"], NORM_EPS, s["o"], s["Wf"], s["Mf"],
                                 s["ws"], int(train))
    else:
        E.e2ttt_chunk_fwd(p, s["q"], s["k"], s["v"], *s["gates"], s["W"], s["M"], s["o"], s["Wf"], s["Mf"], s["ws"], int(train))
    out = {"o": s["o"], "W": s["Wf"], "M": s["Mf"]}
    if not train:
        return out
    if s["normed"]:
        E.e2ttt_chunk_bwd_normed(p, s["q"], s["k"], s["v"], *s["gates"], s["W"], s["M"], s["norm"], NORM_EPS, s["d_o"], None, None,
                                 *s["d_qkv"], *s["d_gates"], s["dW"], s["dM"], s["d_norm"], s["ws"], 1)
        out["d_norm"] = s["d_norm"]
    else:
        E.e2ttt_chunk_bwd(p, s["q"], s["k"], s["v"], *s["gates"], s["W"], s["M"], s["d_o"], None, None, *s["d_qkv"], *s["d_gates"],
                          s["dW"], s["dM"], s["ws"], 1)
    out.update(d_qkv=s["d_qkv"], d_gates=s["d_gates"], dW=s["dW"], dM=s["dM"])
    return out


def work(case):
    """Each input read once, each output written once; products of the method only (nothing recomputed, nothing padded)."""
    B, H, L, d, h = (case[n] for n in ("B", "H", "L", "d", "h"))
    N, nmat, e = B * H, 2 if case["kind"] == "mlp" else 3, 4 if case["io"] == "f32" else 2
    tokens, state = N * L, 4 * N * nmat * d * h
    if case["op"] == "decode":
        return {"bytes": state + 2 * tokens * d * e, "flops": 2 * nmat * d * h * tokens}
    if case["op"] == "prepare":
        return {"bytes": tokens * (4 * d * e + 6 * 4) + tokens * (6 * d * e + 9 * 4), "flops": 40 * tokens * d}
    has_m = case["op"] == "forward" and L <= case["C"]
    nbytes = tokens * (4 * d * e + 12) + state * (4 if has_m else 3)
    # products of a token-head, in units of 2 d h: the network on k and q, the inner backward, two aggregations a matrix
    flops = (2 * nmat + 1 + 2 * nmat) * 2 * d * h * tokens
    if case["op"] == "train":
        nbytes += tokens * (4 * d * e + 12) + 2 * state
        # the adjoints of the outputs, of the aggregations and of the per-token gradients
        flops += (18 if nmat == 2 else 26) * 2 * d * h * tokens
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    if case["op"] == "prepare":
        return {"rel": 4e-3 if case["io"] == "bf16" else 1e-5}
    if case["op"] == "decode":
        return {"rel": 2e-3 if case["io"] == "bf16" else 1e-5}
    if case["io"] == "f32":
        return {"rel": 1e-5}
    # bf16 operands and outputs; the SwiGLU product multiplies its operands' rounding up
    return {"rel": 1e-2 if case["kind"] == "mlp" else 2e-2}
