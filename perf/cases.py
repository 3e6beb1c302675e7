"""The work a program gives to this framework, as cases that can be timed and compared.

A case names one of the public entry points and its sizes:

  op = "decode"    decode_step: one token per sequence, the carried states updated in place
  op = "forward"   chunk_fwd: whole prompts or training batches, fixed length or packed, with or without an initial
                   state, with or without the layer's element-wise operations inside
  op = "train"     chunk_attention under torch.autograd: the forward and every gradient (bf16)
  op = "backward"  chunk_bwd as it is called by default: every gradient, exact, any dtype and head size

B, T, H, dk, dv as in the binding (packed: B = 1, T = all tokens, `seqs` sequences).  Calls are made the way the README
shows them: outputs and workspaces come from the call.
"""
import math

import torch

import paper_2605_05838_b200 as mdn

GATES = ("beta", "log_alpha", "log_mu", "eta")
DTYPES = {"f32": torch.float32, "bf16": torch.bfloat16}


def _case(op, B, T, H, dk=128, dv=128, dtype="bf16", seqs=0, state=False, layer=False):
    return {"op": op, "B": B, "T": T, "H": H, "dk": dk, "dv": dv, "dtype": dtype, "seqs": seqs, "state": state,
            "layer": layer}


def listed():
    cases = {
        # generation for one user: the smallest call there is, latency and launches are all of it
        "decode_one": _case("decode", 1, 1, 16),
        # a server's generation step for a full batch, the layer's element-wise operations inside
        "decode_batch_layer": _case("decode", 128, 1, 16, layer=True),
        # a short follow-up prompt of one user, continued from the state its conversation has reached
        "prefill_short": _case("forward", 1, 200, 16, state=True),
        # the smallest named configuration: fp32, small heads
        "forward_tiny_f32": _case("forward", 1, 256, 2, dk=64, dv=64, dtype="f32"),
        # one layer of the 400M model, a training or evaluation batch
        "forward_400m": _case("forward", 4, 2048, 8),
        # one layer of the 1.3B model, a training or evaluation batch
        "forward_1p3b": _case("forward", 8, 4096, 16),
        # one very long document, continued from a state
        "forward_long": _case("forward", 1, 65536, 16, state=True),
        # prompts of unequal lengths packed into one row
        "forward_packed": _case("forward", 1, 32768, 16, seqs=8),
        # the whole layer (gate formulas, q/k norms, output norm and gate) on a ragged batch
        "forward_layer_ragged": _case("forward", 4, 3001, 16, layer=True),
        # a training step of one layer of the 1.3B model
        "train_1p3b": _case("train", 8, 4096, 16),
        # a training step of one layer of the 400M model on packed documents
        "train_packed_400m": _case("train", 1, 8191, 8, seqs=5),
        # the default backward: exact fp32 gradients
        "backward_f32": _case("backward", 2, 1023, 8, dtype="f32"),
    }
    return [dict(c, name=n) for n, c in cases.items()]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("decode", "decode", "forward", "forward", "packed", "layer", "f32", "train", "train_packed",
                       "backward"))
    H = rng.choice((2, 4, 8, 12, 16, 24, 32))
    if kind == "decode":
        return _case("decode", _log_int(rng, 1, 2048 // H), 1, H, layer=rng.random() < 0.5)
    if kind in ("forward", "layer"):
        B = _log_int(rng, 1, 8)
        T = _log_int(rng, 1 if kind == "forward" else 17, min(65536, (1 << (20 if kind == "forward" else 18)) // (B * H)))
        return _case("forward", B, T, H, state=rng.random() < 0.5, layer=kind == "layer")
    if kind == "packed":
        T = _log_int(rng, 100, (1 << 19) // H)
        return _case("forward", 1, T, H, seqs=_log_int(rng, 2, min(64, T // 16)), state=rng.random() < 0.3)
    if kind == "f32":
        B, H = rng.randint(1, 4), rng.choice((1, 2, 4, 8))
        return _case("forward", B, _log_int(rng, 16, 2048), H, dk=rng.choice((64, 128)), dv=rng.choice((64, 128)),
                     dtype="f32", state=rng.random() < 0.3)
    if kind == "train":
        B = _log_int(rng, 1, 8)
        return _case("train", B, _log_int(rng, 64, min(4096, (1 << 19) // (B * H))), H)
    if kind == "train_packed":
        T = _log_int(rng, 256, min(32768, (1 << 18) // H))
        return _case("train", 1, T, H, seqs=_log_int(rng, 2, min(32, T // 64)))
    B, H = rng.choice(((1, 2), (1, 4), (1, 8), (2, 2), (2, 4), (2, 8), (4, 4)))
    return _case("backward", B, _log_int(rng, 16, 1023), H, dk=rng.choice((64, 128)), dv=rng.choice((64, 128)),
                 dtype=rng.choice(("f32", "f32", "bf16")))


def _gates(g, B, T, H, dk):
    """The stability-aware gate parameterisation on N(0,1) logits, long-memory constants."""
    f32 = dict(device="cuda", dtype=torch.float32, generator=g)
    z = torch.randn((4, B, T, H), **f32)
    eta = torch.tanh(z[3] / math.sqrt(dk)) + 1.0
    theta = torch.atan(eta * 0.25)
    beta = torch.sigmoid(z[0]) * torch.sin(theta) ** 2
    log_alpha = -torch.nn.functional.softplus(z[1] - 4.0) + 2.0 * torch.log(torch.cos(theta))
    log_mu = torch.clamp(-torch.nn.functional.softplus(z[2] - 4.0), min=-1.0)
    return beta, log_alpha, log_mu, eta


def _cuts(g, T, n):
    """cu_seqlens of n sequences of unequal lengths (about 1 : 7 at most) over T tokens."""
    w = torch.rand(n, device="cuda", dtype=torch.float64, generator=g) * 1.5 + 0.25
    cu = torch.zeros(n + 1, device="cuda", dtype=torch.float64)
    cu[1:] = torch.cumsum(w, 0) / w.sum() * T
    cu = torch.round(cu).to(torch.int32)
    cu[n] = T
    return cu


def prepare(case, seed):
    B, T, H, dk, dv = (case[n] for n in ("B", "T", "H", "dk", "dv"))
    dt = DTYPES[case["dtype"]]
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    f32 = dict(device="cuda", dtype=torch.float32, generator=g)

    q, k = torch.randn((B, T, H, dk), **f32), torch.randn((B, T, H, dk), **f32)
    if case["layer"]:   # un-normalised activations, one magnitude per head
        sig = torch.rand((H, 1), **f32) * 1.5 + 0.5
        q, k = q * sig, k * sig
    else:
        q, k = q / q.norm(dim=-1, keepdim=True), k / k.norm(dim=-1, keepdim=True)
    s = {"case": case, "q": q.to(dt), "k": k.to(dt), "v": torch.randn((B, T, H, dv), **f32).to(dt)}
    del q, k
    s["gates"] = _gates(g, B, T, H, dk)

    if case["layer"]:
        x = torch.randn((4, B, T, H), **f32)
        s["gates"] = (x[0], x[1], x[2], 8.0 * x[3])       # the raw projections x_beta, x_alpha, x_mu, x_eta
        s["gate_param"] = dict(a_alpha=torch.rand(H, **f32) * 7.5 + 0.5, b_alpha=0.5 * torch.randn(H, **f32) - 4.0,
                               a_mu=torch.rand(H, **f32) * 7.5 + 0.5, b_mu=0.5 * torch.randn(H, **f32) - 3.0,
                               s=0.25, tau=math.sqrt(2048 / H), log_mu_min=-1.0)
        s["qk_norm"] = dict(d=torch.rand(H, **f32) * 0.7 - 0.2, eps=1e-6)
        s["out_norm_gate"] = dict(g=(1.5 * torch.randn((B, T, H, dv), **f32)).to(dt), w=torch.rand(dv, **f32) + 0.5,
                                  eps=1e-5)

    s["cu"] = _cuts(g, T, case["seqs"]) if case["seqs"] else None
    s["S"] = s["M"] = None
    if case["state"] or case["op"] == "decode":
        n = case["seqs"] or B
        s["S"] = 0.05 * torch.randn((n, H, dk, dv), **f32)
        s["M"] = 0.05 * torch.randn((n, H, dk, dv), **f32)
    if case["op"] in ("train", "backward"):
        s["d_o"] = torch.randn((B, T, H, dv), **f32).to(dt)
    if case["op"] == "train":
        s["leaves"] = [t.detach().requires_grad_() for t in (s["q"], s["k"], s["v"]) + tuple(s["gates"])]
    return s


def run(s):
    op = s["case"]["op"]
    if op == "train":
        o, S, M = mdn.chunk_attention(*s["leaves"], cu_seqlens=s["cu"])
        return (o, S, M) + torch.autograd.grad(o, s["leaves"], s["d_o"])
    if op == "backward":
        return mdn.chunk_bwd(s["q"], s["k"], s["v"], *s["gates"], s["d_o"])
    ops = None
    if s["case"]["layer"]:   # (built for every call: the output gate g is the call's own data)
        ops = mdn.make_layer_ops(s["q"], s["v"], gate_param=s["gate_param"], qk_norm=s["qk_norm"],
                                 out_norm_gate=s["out_norm_gate"])
    if op == "decode":
        return mdn.decode_step(s["q"], s["k"], s["v"], *s["gates"], s["S"], s["M"], layer_ops=ops), s["S"], s["M"]
    return mdn.chunk_fwd(s["q"], s["k"], s["v"], *s["gates"], initial_S=s["S"], initial_M=s["M"], cu_seqlens=s["cu"],
                         layer_ops=ops)


def work(case):
    B, T, H, dk, dv = (case[n] for n in ("B", "T", "H", "dk", "dv"))
    es = 2 if case["dtype"] == "bf16" else 4
    n = B * T * H                                             # head-tokens
    states = 2 * (case["seqs"] or B) * H * dk * dv * 4        # one pair S, M
    qkv, gates = n * (2 * dk + dv) * es, 4 * n * 4
    layer = n * dv * es if case["layer"] else 0               # the output gate g
    if case["op"] == "decode":
        # S^T k, S^T q, and a rank-one update with decay of both states
        return {"bytes": qkv + n * dv * es + gates + layer + 2 * states, "flops": 10.0 * n * dk * dv}
    c = min(64, T)                                            # tokens of a chunk that attend to each other
    # forward, per head-token: K S, K M, Q S, Q M and two state updates; K K^T, Q K^T, T R, W V~ inside the chunk
    fwd_flops = n * (12.0 * dk * dv + 4.0 * c * (dk + dv))
    # backward: the adjoint recurrence (two products, four updates), dO S^T, dO M^T, dR S^T, dR M^T, V~ dS^T, V~ dM^T;
    # W^T dO, T^T dV~, dO V~^T, dR V~^T, and D_W K, D_W^T Q, (D_A + D_A^T) K inside the chunk
    bwd_flops = n * (24.0 * dk * dv + 2.0 * c * (3 * dk + 4 * dv))
    if case["op"] == "forward":
        return {"bytes": qkv + n * dv * es + gates + layer + states * (2 if case["state"] else 1), "flops": fwd_flops}
    if case["op"] == "train":   # q, k, v, gates, dO -> o, S, M, and a gradient for each of the first seven
        return {"bytes": 2 * (qkv + gates) + 2 * n * dv * es + states, "flops": fwd_flops + bwd_flops}
    # backward alone rebuilds the forward's states: K S, K M, two updates, K K^T, Q K^T, T R; fp32 gradients, states' too
    return {"bytes": qkv + gates + n * dv * es + n * (2 * dk + dv) * 4 + gates + states,
            "flops": bwd_flops + n * (8.0 * dk * dv + 2.0 * c * (2 * dk + dv))}


def tolerance(case):
    if case["op"] == "decode":         # fp32 states and arithmetic, one rounding of o to bf16
        return {"rel": 4e-3, "max": 1e-2}
    if case["op"] == "backward":       # fp32 throughout; gate gradients are long sums
        return {"rel": 2e-5, "max": 5e-4}
    if case["dtype"] == "f32":
        return {"rel": 1e-5, "max": 2e-4}
    # bf16 operands of the chunk products, fp32 accumulation
    return {"rel": 1e-2, "max": 1e-1 if case["op"] == "train" else 6e-2}
