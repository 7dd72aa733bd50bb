"""The workloads whose speed counts, and how right their results have to be.

Twelve listed cases, and drawn ones of the same ranges, over the calls that a
DecoMoE serving program makes: decode steps (one token to a batch), prefill
layers from a few hundred tokens to the whole multimodal sequence, the exit
layer, a short stack through the visual exit, attention over the compacted
sequence and over the text-only cache, and the exit gate with the removal that
it triggers. Shapes and distributions are the repository's own synthetic
workloads (48 layers, 128 experts, top 8, hidden 2048, expert width 768, 32
query heads on 4 KV heads of 128).

A case is a dict of plain values whose "kind" says which call it makes:

  layers     one MoE layer call, or the layers of one decode step captured in
             a CUDA graph as a serving loop keeps them
  stack      Stack.forward: RMSNorm and MoE layers through the visual exit
  attention  decomoe_attention: prefill, a chunk over a cache, or a decode step
  exit       the SAVB gate, then the removal of the visual block from the hidden
             state and every layer of both caches, which reads its decision
"""
from __future__ import annotations

import functools
import math

import torch

import paper_2609_38823_gb300 as dm
import workloads as W
from paper_2609_38823_gb300.stack import Stack, StackLayer

D, E, TOPK, M = 2048, 128, 8, 768
HQ, HKV, HD = 32, 4, 128
KV_WIDTH, KV_LAYERS = 512, 48
GATE_H = 512
DEV = "cuda"


def listed():
    return [
        # One token of one sequence: the latency of a decode step, four layers
        # after the exit on the prefix of 64 experts.
        {"name": "decode_T1", "kind": "layers", "T": 1, "K": 64, "zipf": 1.1, "layers": 4, "graph": True},
        # A decode batch of odd size on a wider prefix.
        {"name": "decode_T23", "kind": "layers", "T": 23, "K": 96, "zipf": 1.1, "layers": 4, "graph": True},
        # A larger decode batch (or short prompts) whose prefix the device
        # selects from the routed mass.
        {"name": "layer_T131_mass", "kind": "layers", "T": 131, "K": -1, "p": 0.9, "zipf": 1.1, "layers": 1},
        # The exit layer of a 2048-token prompt: prefix of 64 experts, the
        # 1792 visual rows dropped from its output.
        {"name": "exit_layer_T2048", "kind": "layers", "T": 2048, "K": 64, "zipf": 1.1, "layers": 1, "v0": 0,
         "nv": 1792},
        # A layer before the exit on the longest multimodal sequence: the full
        # pool, the largest call.
        {"name": "layer_T16384", "kind": "layers", "T": 16384, "K": 128, "zipf": 0.8, "layers": 1},
        # The small single-precision layer (reference runs, small models).
        {"name": "layer_f32_T64", "kind": "layers", "T": 64, "K": 10, "f32": True, "layers": 1, "residual": False},
        # Four layers of a prefill through the visual exit: two on the whole
        # 1552-row sequence and the full pool, two on the 272 text rows.
        {"name": "stack_T1552", "kind": "stack", "T": 1552, "v0": 16, "nv": 1280, "layers": 4, "exit": 2, "K": 57},
        # The attention of eight layers of a decode step over the text-only
        # cache that the exit of the longest sequence leaves.
        {"name": "attn_decode_C2049", "kind": "attention", "n": 1, "C": 2049, "calls": 8, "graph": True},
        # Attention of a prefill over a middling sequence, ragged by one row.
        {"name": "attn_prefill_1553", "kind": "attention", "n": 1553, "C": 1553, "calls": 1},
        # Attention of a layer before the exit on the longest sequence.
        {"name": "attn_prefill_16384", "kind": "attention", "n": 16384, "C": 16384, "calls": 1},
        # A follow-up turn: a chunk of new rows over the cache of earlier ones.
        {"name": "attn_chunk_509_4605", "kind": "attention", "n": 509, "C": 4605, "calls": 1},
        # The visual exit after a candidate layer: gate, then removal of 1280
        # visual rows from the hidden state and the 48-layer K and V caches.
        {"name": "exit_T1552", "kind": "exit", "T": 1552, "v0": 16, "nv": 1280},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    pick = rng.choice(["decode", "prefill", "prefill", "f32", "stack", "attn_decode", "attn_prefill", "attn_prefill",
                       "attn_chunk", "exit"])
    if pick == "decode":
        return {"kind": "layers", "T": _log(rng, 1, 48), "K": rng.randint(32, 128), "zipf": rng.choice([0.8, 1.1]),
                "layers": 4, "graph": True}
    if pick == "prefill":
        T = _log(rng, 64, 14000)
        c = {"kind": "layers", "T": T, "zipf": rng.choice([0.8, 1.1, 1.2]), "layers": 1}
        if rng.random() < 0.3:
            c.update(K=-1, p=round(rng.uniform(0.7, 0.98), 3))
        else:
            c.update(K=rng.randint(32, 128))
        if rng.random() < 0.4:
            v0 = rng.randint(0, T // 8)
            c.update(v0=v0, nv=rng.randint(1, T - v0 - 1))
        return c
    if pick == "f32":
        return {"kind": "layers", "T": _log(rng, 1, 300), "K": rng.randint(2, 16), "f32": True, "layers": 1,
                "residual": rng.random() < 0.5}
    if pick == "stack":
        T = _log(rng, 300, 3000)
        v0 = rng.randint(0, 40)
        return {"kind": "stack", "T": T, "v0": v0, "nv": int((T - v0) * rng.uniform(0.4, 0.9)), "layers": 4,
                "exit": rng.randint(1, 3), "K": rng.randint(32, 96)}
    if pick == "attn_decode":
        return {"kind": "attention", "n": rng.randint(1, 8), "C": _log(rng, 64, 16385), "calls": 8, "graph": True}
    if pick == "attn_prefill":
        n = _log(rng, 96, 12000)
        return {"kind": "attention", "n": n, "C": n, "calls": 1}
    if pick == "attn_chunk":
        n = _log(rng, 33, 2048)
        return {"kind": "attention", "n": n, "C": n + _log(rng, 16, 14000), "calls": 1}
    T = _log(rng, 256, 6000)
    v0 = rng.randint(0, 40)
    return {"kind": "exit", "T": T, "v0": v0, "nv": int((T - v0) * rng.uniform(0.4, 0.95))}


def _workload(case):
    if case.get("f32"):
        return W.with_(W.TINY, T=case["T"])
    return W.with_(W.PREFILL, T=case["T"], zipf_s=case.get("zipf", 1.1))


# ------------------------------------------------------------------ inputs

def _layer_inputs(case, seed, layer):
    wl = _workload(case)
    t = W.make_layer(wl, layer=layer, seed=seed, device=DEV)
    if case.get("residual", True):
        t["residual"] = W.make_x(wl, layer=layer, seed=seed, device=DEV, tensor_id=W.TID_RESID)
    return wl, t


def _attention_inputs(case, seed, call):
    g = torch.Generator(device=DEV)
    g.manual_seed(W.stream(seed, 71, call, W.TID_KV))
    shape = lambda rows, heads: torch.randn(rows, heads, HD, generator=g, device=DEV).to(torch.bfloat16)  # noqa: E731
    return shape(case["n"], HQ), shape(case["C"], HKV), shape(case["C"], HKV)


def _exit_inputs(case, seed):
    wl = W.with_(W.STACK, T=case["T"])
    h = W.make_x(wl, seed=seed, device=DEV)
    kv = [W.make_kv(wl, seed=2 * seed + i, device=DEV) for i in range(2)]
    gate = W.make_gate_params(D, GATE_H, [19], 19, seed=seed, device=DEV, margin=4.0)[19]
    return h, kv, gate


def prepare(case, seed):
    kind = case["kind"]
    if kind == "layers":
        return _prepare_layers(case, seed)
    if kind == "stack":
        return _prepare_stack(case, seed)
    if kind == "attention":
        return _prepare_attention(case, seed)
    return _prepare_exit(case, seed)


def _prepare_layers(case, seed):
    calls = []
    ws = None
    for l in range(case["layers"]):
        wl, t = _layer_inputs(case, seed, l)
        dt = dm.DECOMOE_F32 if case.get("f32") else dm.DECOMOE_BF16
        if ws is None:
            ws = dm.workspace(dm.decomoe_moe_layer_workspace_bytes(wl.T, wl.d, wl.E, wl.k, wl.m, dt), DEV)
        w_gu = dm.fuse_gate_up(t.pop("w_gate"), t.pop("w_up"))
        out = torch.empty_like(t["x"])
        kw = {"K_fixed": case["K"], "p": case.get("p", 0.0), "residual": t.get("residual")}
        text = None
        if "nv" in case:
            text = torch.empty(wl.T - case["nv"], wl.d, dtype=t["x"].dtype, device=DEV)
            kw.update(text_out=text, v0=case["v0"], nv=case["nv"])
        calls.append((t["x"], t["w_r"], t["bias"], w_gu, t["w_down"], wl.k, out, ws, kw, text))

    def step():
        for *args, kw, _ in calls:
            dm.decomoe_moe_layer(*args, **kw)

    outs = [o for c in calls for o in ((c[6], c[9]) if c[9] is not None else (c[6],))]
    return _state(case, step, outs)


def _prepare_stack(case, seed):
    wl = _workload(case)
    layers = []
    for l in range(case["layers"]):
        t = W.make_layer(wl, layer=l, seed=seed, device=DEV, with_x=False)
        layers.append(StackLayer(t["w_r"], t["bias"], dm.fuse_gate_up(t["w_gate"], t["w_up"]), t["w_down"]))
        del t
    K = [E] * case["exit"] + [case["K"]] * (case["layers"] - case["exit"])
    st = Stack(layers, K, TOPK, case["exit"], case["v0"], case["nv"], case["T"])
    x = W.make_x(wl, seed=seed, device=DEV)
    return {"step": lambda: st.forward(x), "outs": None}


def _prepare_attention(case, seed):
    ws = dm.workspace(dm.decomoe_attention_workspace_bytes(case["n"], case["C"], HQ, HKV, HD), DEV)
    calls = []
    for i in range(case["calls"]):
        q, k, v = _attention_inputs(case, seed, i)
        calls.append((q, k, v, torch.empty_like(q), ws))

    def step():
        for c in calls:
            dm.decomoe_attention(*c)

    return _state(case, step, [c[3] for c in calls])


def _prepare_exit(case, seed):
    h, kv, gate = _exit_inputs(case, seed)
    left = case["T"] - case["nv"]
    text = torch.empty(left, D, dtype=h.dtype, device=DEV)
    kv_out = [torch.empty(KV_LAYERS, left, KV_WIDTH, dtype=h.dtype, device=DEV) for _ in kv]
    p = torch.zeros(1, device=DEV)
    flag = torch.zeros(1, dtype=torch.int32, device=DEV)
    ws = dm.workspace(dm.decomoe_savb_gate_workspace_bytes(D, GATE_H), DEV)
    v0, nv = case["v0"], case["nv"]

    def step():
        dm.decomoe_savb_gate(h, v0, nv, *gate, 0.5, p, flag, ws)
        dm.decomoe_drop_visual_block_if(flag, h, text, v0, nv)
        for src, dst in zip(kv, kv_out):
            dm.decomoe_drop_visual_block_if(flag, src, dst, v0, nv)

    return {"step": step, "outs": [p, flag, text, *kv_out]}


def _state(case, step, outs):
    if case.get("graph"):
        return {"graph": dm.capture_graph(step), "step": step, "outs": outs}
    return {"step": step, "outs": outs}


def run(state):
    if "graph" in state:
        state["graph"].replay()
        return state["outs"]
    r = state["step"]()
    return state["outs"] if state["outs"] is not None else r


# ------------------------------------------------------------------ work

@functools.lru_cache(maxsize=None)
def _active(T, K, zipf, f32):
    """Experts that the tokens of one layer reach, from one draw of the
    workload's logits."""
    wl = _workload({"T": T, "zipf": zipf, "f32": f32})
    a = W.make_logits(T, wl.E, bias=W._bias(wl), seed=1)
    return int(a[:, :K].topk(wl.k, dim=1).indices.unique().numel())


@functools.lru_cache(maxsize=None)
def _selected(T, p, zipf):
    """The prefix length that the routed mass of one such draw selects."""
    wl = _workload({"T": T, "zipf": zipf})
    v, i = W.make_logits(T, wl.E, bias=W._bias(wl), seed=1).double().topk(wl.k, dim=1)
    mass = torch.zeros(wl.E, dtype=torch.float64).index_add_(0, i.flatten(), v.softmax(1).flatten())
    return max(wl.k, int((mass.cumsum(0) / mass.sum() < p).sum()) + 1)


def _layer_work(T, K, zipf, f32, residual, text):
    wl = _workload({"T": T, "zipf": zipf, "f32": f32})
    e = 4 if f32 else 2
    rows = T * wl.k
    active = _active(T, K, zipf, f32)
    b = active * 3 * wl.m * wl.d * e + wl.E * wl.d * e + (2 + bool(residual)) * T * wl.d * e + text * wl.d * e
    return b, 6 * rows * wl.d * wl.m + 2 * T * wl.d * wl.E


def work(case):
    kind = case["kind"]
    if kind == "layers":
        K = case["K"] if case["K"] > 0 else _selected(case["T"], case["p"], case["zipf"])
        text = case["T"] - case["nv"] if "nv" in case else 0
        b, f = _layer_work(case["T"], K, case.get("zipf", 1.1), case.get("f32", False), case.get("residual", True),
                           text)
        return {"bytes": b * case["layers"], "flops": f * case["layers"]}
    if kind == "stack":
        left = case["T"] - case["nv"]
        got = [_layer_work(case["T"], E, 1.1, False, True, 0)] * case["exit"]
        got += [_layer_work(left, case["K"], 1.1, False, True, 0)] * (case["layers"] - case["exit"])
        return {"bytes": sum(b for b, _ in got), "flops": sum(f for _, f in got)}
    if kind == "attention":
        n, C = case["n"], case["C"]
        seen = n * (C - n) + n * (n + 1) // 2
        return {"bytes": case["calls"] * 2 * HD * (2 * n * HQ + 2 * C * HKV),
                "flops": case["calls"] * 4 * seen * HQ * HD}
    left = case["T"] - case["nv"]
    rows = 2 * KV_LAYERS * KV_WIDTH * left * 2
    return {"bytes": 2 * rows + 2 * 2 * left * D + 4 * GATE_H * (2 * D + 4), "flops": 4 * GATE_H * D}


def tolerance(case):
    """bf16 results: four times the 2.5e-3 by which they are off the 64-bit
    ones (h and the output each rounded to 8 bits; attention's P and output
    likewise). float32: four times the few 1e-7 of the sums over d and m.
    The largest difference is bounded where no routed set can change on a tie
    between logits; whole values and moved rows do not differ."""
    if case["kind"] == "exit":
        return {"rel": 1e-6, "max": 1e-5, "differ": 0.0}
    if case.get("f32"):
        return {"rel": 2e-6, "max": 2e-4}
    if case["kind"] == "attention":
        return {"rel": 1e-2, "max": 0.2}
    return {"rel": 1e-2, "max": 0.9}


# ------------------------------------------------------------------ 64-bit results

def _exact_layer(x, w_r, bias, w_gate, w_up, w_down, k, K, p, residual):
    x = x.double()
    a = x @ w_r.double().T + bias.double()
    if K < 0:
        v, i = a.topk(k, dim=1)
        mass = torch.zeros(a.shape[1], dtype=torch.float64, device=x.device)
        mass.index_add_(0, i.flatten(), v.softmax(1).flatten())
        K = max(k, int((mass.cumsum(0) / mass.sum() < p).sum()) + 1)
    v, i = a[:, :K].topk(k, dim=1)
    w = v.softmax(1)
    out = torch.zeros_like(x) if residual is None else residual.double()
    for e in range(K):
        t, j = (i == e).nonzero(as_tuple=True)
        if t.numel():
            r = x[t]
            h = torch.nn.functional.silu(r @ w_gate[e].double().T) * (r @ w_up[e].double().T)
            out.index_add_(0, t, w[t, j][:, None] * (h @ w_down[e].double().T))
    return out


def _text(out, v0, nv):
    return torch.cat([out[:v0], out[v0 + nv:]])


def exact(case, seed):
    kind = case["kind"]
    if kind == "layers":
        outs = []
        for l in range(case["layers"]):
            wl, t = _layer_inputs(case, seed, l)
            o = _exact_layer(t["x"], t["w_r"], t["bias"], t["w_gate"], t["w_up"], t["w_down"], wl.k, case["K"],
                             case.get("p", 0.0), t.get("residual"))
            outs += [o, _text(o, case["v0"], case["nv"])] if "nv" in case else [o]
        return outs
    if kind == "stack":
        wl = _workload(case)
        h = W.make_x(wl, seed=seed, device=DEV).double()
        for l in range(case["layers"]):
            if l == case["exit"]:
                h = _text(h, case["v0"], case["nv"])
            t = W.make_layer(wl, layer=l, seed=seed, device=DEV, with_x=False)
            K = E if l < case["exit"] else case["K"]
            n = h * torch.rsqrt(h.square().mean(1, keepdim=True) + 1e-6)
            h = _exact_layer(n, t["w_r"], t["bias"], t["w_gate"], t["w_up"], t["w_down"], TOPK, K, 0.0, h)
        return h
    if kind == "attention":
        return [_exact_attention(*_attention_inputs(case, seed, i)) for i in range(case["calls"])]
    h, kv, (w1, b1, w2, b2) = _exit_inputs(case, seed)
    text = _text(h, case["v0"], case["nv"]).double()
    x = torch.cat([text[:-1].mean(0), text[-1]])
    z = w2.double() @ (w1.double() @ x + b1.double()).relu() + b2.double()
    p = z.softmax(0)[1:]
    left = [torch.cat([c[:, :case["v0"]], c[:, case["v0"] + case["nv"]:]], 1).double() for c in kv]
    return [p, None, text, *left]


def _exact_attention(q, k, v):
    n, C = q.shape[0], k.shape[0]
    out = torch.empty(n, HQ, HD, dtype=torch.float64, device=q.device)
    cols = torch.arange(C, device=q.device)
    for head in range(HQ):
        kh, vh = k[:, head // (HQ // HKV)].double(), v[:, head // (HQ // HKV)].double()
        for r0 in range(0, n, 4096):
            r1 = min(n, r0 + 4096)
            last = C - n + r1
            s = q[r0:r1, head].double() @ kh[:last].T / math.sqrt(HD)
            s.masked_fill_(cols[None, :last] > (C - n + torch.arange(r0, r1, device=q.device))[:, None], -math.inf)
            out[r0:r1, head] = s.softmax(1) @ vh[:last]
    return out
