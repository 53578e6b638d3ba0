"""Performance cases of the MoE-FFN layer: what a program that uses this framework calls, over the sizes it calls it with.

A case is a dict of plain values.  `path` says which calls a pass makes, the rest are sizes and options:

  infer       scores of the tokens (`gate_input`: "x" = the router in the path, "logits" = logits the program already has),
              then the forward layer
  train       the same, then the backward layer into the program's gradient buffers
  host_train  one training step whose activations live in pinned host memory (the *_host calls)
  router      the router in the path, forward, and the score gradient of an earlier micro-batch
  layout      routing and the dispatch layout alone, without a context's workspace (programs that bring their own expert kernels)
  ep          expert-parallel dispatch and combine with every rank of the group on this GPU

T tokens, T_max the context's capacity, d hidden size, E routed experts, k per token, S shared experts, F expert intermediate
size; `gate` softmax or sigmoid, `renorm` the k scores; `zipf` > 0 skews the experts' popularity and leaves four experts empty.
"""
import math

import numpy as np
import torch

from paper_2605_23764_b200 import MoeLayer
from paper_2605_23764_b200 import binding as B

BF16 = torch.bfloat16
EP_FFN = 128   # the ep path's contexts only route and lay out: their F is not used


def _case(path, T, d, E, k, S, F, **more):
    c = {"path": path, "T": T, "T_max": T, "d": d, "E": E, "k": k, "S": S, "F": F, "gate": "softmax", "renorm": True,
         "gate_input": "logits", "zipf": 0.0, "ranks": 1}
    c.update(more)
    return c


def listed():
    named = [
        # token generation, a few sequences in flight, V2-Lite-shaped layer: bound by the weights of the experts that are hit and by latency
        ("decode_lite_8", _case("infer", 8, 2048, 64, 6, 2, 1408, T_max=256, gate_input="x", renorm=False)),
        # token generation, a serving batch, V3-shaped layer: most experts are hit by one or two tokens each
        ("decode_v3_64", _case("infer", 64, 7168, 256, 8, 1, 2048, T_max=256, gate_input="x")),
        # prompt processing, V2-Lite-shaped layer (workloads/configs.py, configuration 1)
        ("prefill_lite_4096", _case("infer", 4096, 2048, 64, 6, 2, 1408, renorm=False)),
        # prompt processing, V3-shaped layer (configuration 2)
        ("prefill_v3_4096", _case("infer", 4096, 7168, 256, 8, 1, 2048)),
        # prompt processing, skewed expert popularity with empty experts (configuration 3)
        ("prefill_zipf_16384", _case("infer", 16384, 4096, 128, 8, 0, 1536, zipf=1.2)),
        # the smallest training step (configuration 0): launches and host time
        ("train_tiny_256", _case("train", 256, 256, 8, 2, 0, 128)),
        # a training step of the V3-shaped layer at 256 rows an expert: one half of configuration 4
        ("train_v3_4096", _case("train", 4096, 7168, 128, 8, 0, 2048)),
        # a training step with sizes that fit no tile (tokens, hidden, intermediate), sigmoid scores, a shared expert
        ("train_ragged_1777", _case("train", 1777, 1160, 24, 3, 1, 712, gate="sigmoid")),
        # a training step fed from pinned host memory, V2-Lite-shaped experts: the end-to-end call of a host-side loop
        ("host_train_lite_4096", _case("host_train", 4096, 2048, 64, 6, 0, 1408, renorm=False)),
        # the router of a V3-shaped training step, both directions
        ("router_v3_8192", _case("router", 8192, 7168, 256, 8, 0, 2048)),
        # routing and layout of a serving step that runs its own expert kernels: the smallest calls
        ("layout_1024", _case("layout", 1024, 2048, 64, 6, 2, 1408, renorm=False)),
        # the token exchange of an expert-parallel group of eight, tokens of configuration 4
        ("ep_8192", _case("ep", 8192, 7168, 256, 8, 0, EP_FFN, ranks=8)),
    ]
    return [dict(c, name=n) for n, c in named]


# ---------------------------------------------------------------- what a pass cannot do without
def _experts_hit(c):
    """Expected number of routed experts that receive a token."""
    if c["zipf"]:
        p = [(r + 1.0) ** -c["zipf"] for r in range(c["E"] - 4)]
        tot = sum(p)
        return sum(1.0 - (1.0 - min(1.0, c["k"] * v / tot)) ** c["T"] for v in p)
    return c["E"] * (1.0 - (1.0 - c["k"] / c["E"]) ** c["T"])


def work(case):
    T, d, E, k, S, F = (case[n] for n in ("T", "d", "E", "k", "S", "F"))
    act, scores, rows = 2.0 * T * d, 8.0 * T * k, T * (k + S)
    if case["path"] == "layout":
        return {"bytes": 4.0 * T * E + scores + 8.0 * rows + 8.0 * (E + S), "flops": 0.0}
    if case["path"] == "router":   # forward: x, W_r -> logits and scores; backward: logits, ids, gradient -> gradient
        return {"bytes": act + 2.0 * E * d + 4.0 * T * E + scores + 8.0 * T * E + scores, "flops": 2.0 * T * E * d}
    if case["path"] == "ep":       # dispatch: x -> rows and their meta; combine: rows -> returned rows -> sums
        return {"bytes": act + 2.0 * rows * d + 16.0 * rows + 3 * 2.0 * rows * d + act, "flops": 0.0}
    hit = _experts_hit(case) + S
    weights = 6.0 * d * F
    gate = 2.0 * E * d if case["gate_input"] == "x" else 4.0 * T * E
    gate_flops = 2.0 * T * E * d if case["gate_input"] == "x" else 0.0
    fwd_bytes, fwd_flops = gate + scores + 2 * act + hit * weights, 6.0 * rows * d * F
    if case["path"] == "infer":
        return {"bytes": fwd_bytes, "flops": fwd_flops + gate_flops}
    # each of the two calls reads the weights; every gradient slab is written
    bwd_bytes = 2 * act + 4.0 * T * k + hit * weights + (E + S) * weights
    return {"bytes": fwd_bytes + bwd_bytes, "flops": 3 * fwd_flops + gate_flops}


def _cost(case):
    w = work(case)
    return max(w["bytes"], w["flops"] / 50)


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """A case of the same paths, its sizes spread over the listed ranges; never dearer than the dearest listed case."""
    most = max(_cost(c) for c in listed())
    while True:
        path = rng.choice(["infer", "infer", "infer", "train", "train", "host_train", "router", "layout", "ep"])
        d = 8 * _log_int(rng, 32, 896)
        E = rng.choice([8, 16, 24, 32, 40, 64, 100, 128, 160, 256])
        k = rng.randint(1, min(8, E))
        c = _case(path, 0, d, E, k, 0, 0, gate=rng.choice(["softmax", "softmax", "sigmoid"]), renorm=rng.random() < 0.7)
        if path in ("infer", "train", "host_train"):
            # three expert sizes in four are multiples of 16, as model configurations have them
            c["F"] = 16 * _log_int(rng, 8, 128) if rng.random() < 0.75 else 8 * (2 * _log_int(rng, 8, 128) - 1)
            c["S"] = rng.choice([0, 0, 1, 2])
        else:
            c["F"] = EP_FFN
        if path == "infer":
            c["T"] = _log_int(rng, 1, 16384)
            c["T_max"] = c["T"] if c["T"] >= 1024 else max(c["T"], 256)
            c["gate_input"] = rng.choice(["x", "logits"])
            if c["gate_input"] == "logits" and E >= 16 and k <= E - 4 and rng.random() < 0.3:
                c["zipf"] = round(rng.uniform(0.6, 1.2), 2)
        elif path == "train":
            c["T"] = c["T_max"] = _log_int(rng, 64, 8192)
        elif path == "host_train":
            c["T"] = c["T_max"] = _log_int(rng, 256, 4096)
        elif path == "router":
            c["T"] = c["T_max"] = _log_int(rng, 16, 16384)
        elif path == "layout":
            c["T"] = c["T_max"] = _log_int(rng, 16, 16384)
            c["S"] = rng.choice([0, 1, 2])
        else:
            c["ranks"] = rng.choice([r for r in (2, 4, 8) if E % r == 0])
            c["T"] = c["T_max"] = _log_int(rng, 512, 8192)
        # the dearest case bounds the time; the gradient slabs bound the memory
        if _cost(c) <= most and c["T"] * (k + c["S"]) <= 131072 and 3.0 * (E + c["S"]) * d * c["F"] <= 11.4e9 / (
                1 if path == "infer" else 2):
            return c


# ---------------------------------------------------------------- what a program has in hand
def _normal(gen, shape, std, dtype=BF16):
    return torch.empty(shape, dtype=dtype, device="cuda").normal_(0.0, std, generator=gen)


def _logits(gen, c, T):
    """Router logits as x.W_r gives them with x ~ N(0, 1), W_r ~ N(0, std 0.02), plus the popularity bias."""
    logits = _normal(gen, (T, c["E"]), 0.02 * math.sqrt(c["d"]), torch.float32)
    if c["zipf"]:
        rank = torch.randperm(c["E"], generator=gen, device="cuda").to(torch.float32)
        bias = -c["zipf"] * torch.log(rank + 1.0)
        bias[rank >= c["E"] - 4] = -1.0e4
        logits += bias
    return logits


def _layer(c, **more):
    return MoeLayer(c["T_max"], c["d"], c["E"], c["k"], c["S"], c["F"], renorm=c["renorm"],
                    sigmoid_gate=c["gate"] == "sigmoid", **more)


def prepare(case, seed):
    c = case
    T, d, E, k, S, F = (c[n] for n in ("T", "d", "E", "k", "S", "F"))
    gen = torch.Generator(device="cuda").manual_seed(seed)
    s = {"c": c}
    if c["path"] == "ep":
        return _prepare_ep(s, gen)
    if c["path"] == "layout":
        s["layer"] = _layer(c)
        s["logits"] = _logits(gen, c, T)
        return s
    x = _normal(gen, (T, d), 1.0)
    if c["path"] == "router":
        s["layer"] = _layer(c)
        s["x"], s["W_r"] = x, _normal(gen, (E, d), 0.02)
        # the earlier micro-batch whose gradient arrives: its logits, selection and score gradient
        s["old_logits"] = _logits(gen, c, T)
        s["old_ids"] = torch.topk(s["old_logits"], k, dim=1).indices.to(torch.int32).contiguous()
        s["d_topk_w"] = _normal(gen, (T, k), 1.0, torch.float32)
        return s
    s["layer"] = _layer(c, save_for_bwd=c["path"] != "infer")
    s["W_gate_up"] = _normal(gen, (E + S, 2 * F, d), d ** -0.5)
    s["W_down"] = _normal(gen, (E + S, d, F), d ** -0.5)
    if c["gate_input"] == "x":
        s["W_r"] = _normal(gen, (E, d), 0.02)
    else:
        s["logits"] = _logits(gen, c, T)
    s["x"] = x
    if c["path"] != "infer":
        s["dout"] = _normal(gen, (T, d), 1.0)
        s["dW_gate_up"], s["dW_down"] = torch.empty_like(s["W_gate_up"]), torch.empty_like(s["W_down"])
    if c["path"] == "host_train":
        for n in ("x", "logits", "dout"):
            s[n] = s[n].cpu().pin_memory()
        pinned = dict(device="cpu", pin_memory=True)
        s["ids"] = torch.empty(T, k, dtype=torch.int32, **pinned)
        s["w"] = torch.empty(T, k, dtype=torch.float32, **pinned)
        s["d_w"] = torch.empty(T, k, dtype=torch.float32, **pinned)
        s["out"], s["dx"] = torch.empty(T, d, dtype=BF16, **pinned), torch.empty(T, d, dtype=BF16, **pinned)
    return s


def _prepare_ep(s, gen):
    """Tokens spread evenly over the ranks (the first ones take the remainder), routed and laid out rank by rank; the
    plans come from the gathered counts, as in a group of processes."""
    c = s["c"]
    T, d, E, k, R = (c[n] for n in ("T", "d", "E", "k", "ranks"))
    Ts = [T // R + (r < T % R) for r in range(R)]
    i32 = dict(dtype=torch.int32, device="cuda")
    layer = MoeLayer(max(Ts), d, E, k, 0, c["F"], renorm=c["renorm"], sigmoid_gate=c["gate"] == "sigmoid")
    xs, ws, src, counts = [], [], [], []
    for Tr in Ts:
        xs.append(_normal(gen, (Tr, d), 1.0))
        ids, w = layer.route(_logits(gen, c, Tr))
        cnt, _, _, src_of = layer.layout(ids)
        ws.append(w)
        src.append(src_of)
        counts.append(cnt)
    counts = torch.stack(counts).cpu().numpy().astype(np.int32)
    plans = [B.moe_ep_plan(counts, r) for r in range(R)]
    rows = [int(n) for n in plans[0][1]]
    layer.close()
    # every rank's receive buffer is a piece of one allocation (a rank may receive nothing: its pointer still has to be valid)
    first = [sum(rows[:r]) for r in range(R)]
    all_recv, all_meta = torch.empty(T * k + 1, d, dtype=BF16, device="cuda"), torch.empty(T * k + 1, 4, **i32)
    recv = [all_recv[first[r]:first[r] + max(rows[r], 1)] for r in range(R)]
    meta = [all_meta[first[r]:first[r] + max(rows[r], 1)] for r in range(R)]
    ret = [torch.empty(Tr * k, d, dtype=BF16, device="cuda") for Tr in Ts]
    recv_cnt = [torch.zeros(max(-(-n // B.MOE_EP_BLOCK_ROWS), 1), **i32) for n in rows]
    ret_cnt = [torch.zeros(max(-(-Tr // B.MOE_EP_TOKEN_BLOCK), 1), **i32) for Tr in Ts]
    tickets = [torch.zeros(2, **i32) for _ in range(R)]
    tasks = [torch.from_numpy(p[0]).cuda() if len(p[0]) else None for p in plans]
    out = [torch.empty(Tr, d, dtype=BF16, device="cuda") for Tr in Ts]
    y = [_normal(gen, (max(n, 1), d), 1.0) for n in rows]   # what the experts made of the received rows
    s["peers"] = [B.moe_ep_peer(recv[r], meta[r], recv_cnt[r], ret[r], ret_cnt[r]) for r in range(R)]
    s["dispatch"] = [dict(rank=r, T=Ts[r], x=xs[r], topk_w=ws[r], src_of=src[r], tasks=tasks[r], recv_rows=rows[r],
                          consumed=None, ticket=tickets[r]) for r in range(R)]
    s["combine"] = [dict(rank=r, T=Ts[r], recv_rows=rows[r], y=y[r], out=out[r], ticket=tickets[r]) for r in range(R)]
    s["status"] = torch.zeros(4, **i32)
    s["keep"] = (recv_cnt, ret, ret_cnt)
    s["recv"], s["meta"], s["out"] = all_recv[:T * k], all_meta[:T * k], out
    return s


# ---------------------------------------------------------------- one pass
def run(s):
    c = s["c"]
    T, E, k, S = c["T"], c["E"], c["k"], c["S"]
    path = c["path"]
    i32 = dict(dtype=torch.int32, device="cuda")
    if path == "ep":
        B.moe_ep_dispatch(s["peers"], s["dispatch"], k, c["d"], s["status"])
        B.moe_ep_combine(s["peers"], s["combine"], k, c["d"], s["status"])
        return [s["recv"], s["meta"], s["status"]] + s["out"]
    layer = s["layer"]
    if path == "layout":
        ids, w = layer.route(s["logits"])
        counts, offsets = torch.empty(E + S, **i32), torch.empty(E + S + 1, **i32)
        row_of, src_of = torch.empty(T * (k + S), **i32), torch.empty(T * (k + S), **i32)
        B.moe_layout_noalloc(ids, T, E, k, S, counts, offsets, row_of, src_of)
        return ids, w, counts, offsets, row_of, src_of
    if path == "host_train":
        B.moe_route_host(layer.ctx, s["logits"], T, s["ids"], s["w"])
        B.moe_ffn_fwd_host(layer.ctx, s["x"], s["ids"], s["w"], s["W_gate_up"], s["W_down"], s["out"], T)
        B.moe_ffn_bwd_host(layer.ctx, s["dout"], s["W_gate_up"], s["W_down"], s["dx"], s["dW_gate_up"], s["dW_down"],
                           s["d_w"], T)
        return s["ids"], s["w"], s["out"], s["dx"], s["d_w"], s["dW_gate_up"], s["dW_down"]
    if path == "router" or c["gate_input"] == "x":
        ids = torch.empty(T, k, **i32)
        w = torch.empty(T, k, dtype=torch.float32, device="cuda")
        logits = torch.empty(T, E, dtype=torch.float32, device="cuda") if path == "router" else None
        B.moe_router_fwd(layer.ctx, s["x"], s["W_r"], T, ids, w, logits)
        if path == "router":
            d_logits = torch.empty(T, E, dtype=torch.float32, device="cuda")
            B.moe_router_bwd(layer.ctx, s["old_logits"], s["old_ids"], s["d_topk_w"], T, d_logits)
            return ids, w, logits, d_logits
    else:
        ids, w = layer.route(s["logits"])
    out = layer.ffn_fwd(s["x"], ids, w, s["W_gate_up"], s["W_down"])
    if path == "infer":
        return ids, w, out
    dx, _, _, d_w = layer.ffn_bwd(s["dout"], s["x"], ids, w, s["W_gate_up"], s["W_down"],
                                  dW_gate_up=s["dW_gate_up"], dW_down=s["dW_down"])
    return ids, w, out, dx, d_w, s["dW_gate_up"], s["dW_down"]


def tolerance(case):
    if case["path"] == "layout":   # integers the same; scores are fp32 exponentials
        return {"rel": 1e-5, "max": 1e-4}
    if case["path"] == "router":   # fp32 sums of bf16 products; logits nearer to each other than their rounding may swap places
        return {"rel": 1e-5, "max": 1e-3, "differ": 1e-3}
    if case["path"] == "ep":       # rows are copied, sums are rounded to bf16 once
        return {"rel": 5e-3, "max": 2e-2}
    # bf16 operands, fp32 sums, bf16 results; a logit of the in-path router may be rounded the other way at a tie
    return {"rel": 1e-2, "differ": 2e-3 if case["gate_input"] == "x" else 0.0}
