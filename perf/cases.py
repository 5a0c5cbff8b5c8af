"""The layer calls that this framework's users make, as measurable cases.

A case is one use of ``pmpe.MoeLayer`` (or of a stack of layers): the layer's
shape, the number of tokens, how the tokens divide into authorised (ALLOW) and
other requests, and the call: a forward as a serving step makes it, or one of
the training steps (forward and a backward).  Shapes are those of
``configs.CONFIGS`` and of the paper's own private pools (16 experts, top-8);
weights, hidden states and router skew follow ``inputs``.

Calls (``mode``):
  forward     serving: the layer alone, with its route log
  serve       serving with metadata and audit: per-token policy bytes from the
              requests' bytes and offsets, the audit reset, the layer with its
              route log and audit counters
  stack       ``layers`` decoder layers one after another, residual add between
  train       forward, then the private gradients and the input gradient in one
              pass (a wrapped layer with trained layers below it); ``saved``: the
              forward keeps its gate/up accumulators for the backward
  private     forward, then the private gradients alone (the lowest trained layer)
  input       forward, then the input gradient alone (a frozen layer above
              trained ones)
"""
from __future__ import annotations

import math

import torch

from paper_2608_06690_gb300 import inputs as inp
from paper_2608_06690_gb300 import pmpe
from paper_2608_06690_gb300.configs import CONFIGS
from paper_2608_06690_gb300.inputs import LayerShape

LAYERS = {
    "tiny": dict(H=256, I=128, E_pub=16, E_priv=4, E_sh=0, k=2, renorm=True, skew=False),
    "qwen3": dict(H=2048, I=768, E_pub=128, E_priv=32, E_sh=0, k=8, renorm=True, skew=False),
    "qwen3_16priv": dict(H=2048, I=768, E_pub=128, E_priv=16, E_sh=0, k=8, renorm=True, skew=False),
    "deepseek": dict(H=2048, I=1408, E_pub=64, E_priv=16, E_sh=2, k=6, renorm=False, skew=True),
}
SKEW = CONFIGS["deepseek_v2_lite"].skew


def _case(layer, mode, T, requests, allow, **more):
    return dict(LAYERS[layer], mode=mode, T=T, requests=requests, allow=allow, layers=1, saved=False, **more)


def listed():
    cases = [
        # the smallest layer, one token a request: all latency and launches
        dict(_case("tiny", "forward", 64, 64, 0.5), name="tiny_t64"),
        # one user's decode step: a single authorised token, eight experts' weights
        dict(_case("qwen3", "forward", 1, 1, 1.0), name="qwen3_decode_t1"),
        # a decode batch of 64 users, half of them authorised
        dict(_case("qwen3", "forward", 64, 64, 0.5), name="qwen3_decode_t64"),
        # a decode batch on the layer with shared experts and the pool softmax
        dict(_case("deepseek", "forward", 96, 96, 0.25), name="deepseek_decode_t96"),
        # decoder layers in sequence, as a model runs them in one decode step
        dict(_case("qwen3", "stack", 37, 37, 0.5), name="qwen3_stack4_t37", layers=4),
        # a serving step that mixes ragged prompt chunks with decode tokens, with
        # per-request policies expanded on the device and the audit kept
        dict(_case("qwen3", "serve", 777, 23, 0.5), name="qwen3_mixed_t777"),
        # prompt processing: 16 requests, half authorised, audited
        dict(_case("qwen3", "serve", 4096, 16, 0.5), name="qwen3_prefill_t4096"),
        # prompt processing of the skewed layer with shared experts
        dict(_case("deepseek", "forward", 8192, 32, 0.25), name="deepseek_prefill_t8192"),
        # a large prompt batch, one layer of the 48-layer stack
        dict(_case("qwen3", "forward", 16384, 64, 0.5), name="qwen3_prefill_t16384"),
        # a training step of a wrapped layer, gate/up accumulators saved
        dict(_case("qwen3", "train", 4096, 16, 0.5), name="qwen3_train_t4096", saved=True),
        # the lowest trained layer: private gradients only, an odd batch, the paper's pool of 16
        dict(_case("qwen3_16priv", "private", 1000, 7, 0.5), name="qwen3_private_t1000"),
        # a layer passing its gradient down, recomputing, shared experts and pool softmax
        dict(_case("deepseek", "train", 3000, 11, 0.25), name="deepseek_train_t3000"),
    ]
    return cases


def draw(rng):
    """The same layers and small generic ones, tokens over their whole range
    (by logarithm), ragged requests, every call."""
    kind = rng.choice(["qwen3", "qwen3", "qwen3_16priv", "deepseek", "deepseek", "generic"])
    mode = rng.choice(["forward", "forward", "serve", "stack", "train", "private", "input"])
    if kind == "generic":
        k = rng.choice([1, 2, 4, 6, 8])
        dims = dict(H=128 * rng.randint(1, 12), I=128 * rng.randint(1, 8), E_pub=rng.randint(max(k, 8), 128),
                    E_priv=rng.randint(max(k, 4), 48), E_sh=rng.choice([0, 0, 1, 2]), k=k, renorm=rng.random() < 0.6,
                    skew=False)
    else:
        dims = dict(LAYERS[kind])
    most = {"forward": 16384, "serve": 16384, "stack": 512, "train": 4096, "private": 4096, "input": 4096}[mode]
    if kind == "deepseek":
        most = min(most, 8192 if mode in ("forward", "serve") else (512 if mode == "stack" else 3000))
    T = int(round(math.exp(rng.uniform(0.0, math.log(most)))))
    requests = max(1, min(T, int(round(math.exp(rng.uniform(0.0, math.log(64.0)))))))
    case = dict(dims, mode=mode, T=T, requests=requests, allow=rng.choice([0.0, 0.25, 0.5, 0.5, 0.75, 1.0]),
                layers=rng.randint(2, 4) if mode == "stack" else 1,
                saved=mode in ("train", "private", "input") and rng.random() < 0.5)
    return case


def _shape(case):
    return LayerShape(case["T"], case["H"], case["I"], case["E_pub"], case["E_priv"], case["E_sh"], case["k"],
                      bool(case["renorm"]))


def _requests(case, seed):
    """One policy byte per request and the requests' cumulative offsets: ragged
    contiguous spans; ALLOW requests spread evenly in number."""
    g = torch.Generator().manual_seed(int(seed) + 71)
    T, n = case["T"], case["requests"]
    cuts = torch.sort(torch.randperm(T - 1, generator=g)[:n - 1] + 1).values if n > 1 else torch.zeros(0, dtype=torch.int64)
    cu = torch.cat([torch.zeros(1, dtype=torch.int64), cuts, torch.tensor([T])]).to(torch.int32)
    byte = torch.zeros(n, dtype=torch.uint8)
    byte[torch.randperm(n, generator=g)[:int(round(case["allow"] * n))]] = inp.ALLOW
    return byte, cu


def _inputs(case, seed, layer=0):
    s = _shape(case)
    skew = SKEW if case["skew"] else None
    return inp.make_weights(s, int(seed) * 64 + layer, device="cuda", skew=skew)


def _hidden(case, seed):
    return inp.make_hidden(_shape(case), int(seed), device="cuda", skew=SKEW if case["skew"] else None)


def _dout(case, seed):
    g = torch.Generator(device="cuda").manual_seed(int(seed) + 97)
    return torch.randn((case["T"], case["H"]), generator=g, device="cuda").to(torch.bfloat16)


def prepare(case, seed):
    s = _shape(case)
    ws = pmpe.Workspace("cuda")  # layers run in sequence share one scratch buffer
    layers = [pmpe.MoeLayer(s, _inputs(case, seed, l), workspace=ws) for l in range(case["layers"])]
    byte, cu = _requests(case, seed)
    policy = byte.repeat_interleave((cu[1:] - cu[:-1]).long()).cuda()
    st = dict(case=case, layers=layers, hidden=_hidden(case, seed), policy=policy, byte=byte.cuda(), cu=cu.cuda(),
              idx=torch.empty((s.T, s.k), dtype=torch.int32, device="cuda"),
              w=torch.empty((s.T, s.k), dtype=torch.float32, device="cuda"))
    if case["mode"] == "serve":
        st["audit"] = torch.zeros(pmpe.audit_words(s.T, s.E), dtype=torch.int32, device="cuda")
    if case["mode"] in ("train", "private", "input"):
        st["dout"] = _dout(case, seed)
    return st


def run(st):
    case, layer, h, policy = st["case"], st["layers"][0], st["hidden"], st["policy"]
    mode, T = case["mode"], case["T"]
    if mode == "stack":
        x = h
        for lay in st["layers"]:
            x = x + lay.forward(x, policy)
        return x
    if mode == "forward":
        out = layer.forward(h, policy, topk_idx=st["idx"], topk_w=st["w"])
        return {"out": out, "idx": st["idx"], "w": st["w"]}
    if mode == "serve":
        E = case["E_pub"] + case["E_priv"]
        pol = pmpe.policy_from_requests(st["byte"], st["cu"], T)
        pmpe.audit_reset(st["audit"], T, E)
        out = layer.forward(h, pol, topk_idx=st["idx"], topk_w=st["w"], audit=st["audit"])
        return {"out": out, "idx": st["idx"], "w": st["w"], "policy": pol, "audit": st["audit"]}
    out = layer.forward(h, policy, save_for_backward=case["saved"])
    if mode == "private":
        return {"out": out, "grads": layer.backward_private(h, policy, st["dout"])}
    if mode == "input":
        return {"out": out, "d_hidden": layer.backward_input(h, policy, st["dout"])}
    grads, d_hidden = layer.backward(h, policy, st["dout"])
    return {"out": out, "grads": grads, "d_hidden": d_hidden}


def _touched(E, k, n):
    """Experts of a pool that n tokens reach, each with k of E (even load)."""
    return E * (1.0 - (1.0 - k / E) ** n) if n > 0 else 0.0


def work(case):
    """Every input read once and every result written once; the multiplications
    of the layer's own GEMMs (no recomputation in a backward)."""
    T, H, I, k = case["T"], case["H"], case["I"], case["k"]
    n = case["requests"]
    na = T * int(round(case["allow"] * n)) / n  # ALLOW tokens: requests of even length on average
    nd = T - na
    experts = _touched(case["E_pub"], k, nd) + _touched(case["E_priv"], k, na) + case["E_sh"]
    rows = T * (k + case["E_sh"])
    router = (case["E_pub"] if nd else 0) + (case["E_priv"] if na else 0)
    w_bytes = (experts * 3 * I * H + router * H) * 2
    r_flops = 2 * H * (nd * case["E_pub"] + na * case["E_priv"])
    n_bytes = w_bytes + T * H * 2 + T * H * 2 + T
    flops = rows * 6 * H * I + r_flops
    mode = case["mode"]
    if mode in ("forward", "serve"):
        n_bytes += T * k * 8
    if mode == "serve":
        n_bytes += 4 * (2 + 3 * (case["E_pub"] + case["E_priv"]) + 2 * T) + 5 * n
    if mode == "stack":
        n_bytes = case["layers"] * w_bytes + T * H * 4 + T
        flops *= case["layers"]
    if mode in ("train", "private", "input"):
        n_bytes += T * H * 2
        priv = na * k
        if mode != "input":
            n_bytes += 4 * case["E_priv"] * (3 * I * H + H)
            flops += priv * 6 * H * I + na * 2 * H * case["E_priv"]
        if mode == "private":
            flops += priv * 2 * H * I
        else:
            n_bytes += T * H * 4
            flops += rows * 6 * H * I + r_flops
    return {"bytes": float(n_bytes), "flops": float(flops)}


def tolerance(case):
    """Activations, per-row outputs and the result are BF16 (2^-9 each): outputs
    and gradients are 2.3e-3 to 2.9e-3 off the 64-bit result, the stack, whose
    later layers route on rounded states, 0.7e-2 to 1.1e-2; about four times
    that.  Tokens whose k-th and next logits agree to FP32 rounding may take
    another expert in another order of summation (a few in 10^5): their rows
    differ by the order of the result itself, which ``max`` and ``differ`` leave
    room for."""
    return {"rel": 3e-2 if case["mode"] == "stack" else 1.2e-2, "max": 0.9, "differ": 0.01}


# ------------------------------------------------------------ the same in 64 bits

def _layer64(case, w, h, policy, dout=None, need_w=False, need_h=False):
    """One layer in FP64: (out, idx, weights, gradients, input gradient)."""
    k, E_pub = case["k"], case["E_pub"]
    h64 = h.double()
    T = h.shape[0]
    out = torch.zeros_like(h64)
    dh = torch.zeros_like(h64)
    idx = torch.empty((T, k), dtype=torch.int32, device=h.device)
    wts = torch.empty((T, k), dtype=torch.float64, device=h.device)
    grads = None
    if need_w:
        E, I, H = case["E_priv"], case["I"], case["H"]
        f8 = dict(dtype=torch.float64, device=h.device)
        grads = {"d_router": torch.zeros((E, H), **f8), "d_gate": torch.zeros((E, I, H), **f8),
                 "d_up": torch.zeros((E, I, H), **f8), "d_down": torch.zeros((E, H, I), **f8)}
    d64 = dout.double() if dout is not None else None
    allowed = policy == inp.ALLOW

    def expert(tok, wt, wg, wu, wd):
        """Output of the rows and, with dout, (dL/dw, dA, dG, dU, w act)."""
        a_in = h64[tok]
        g, u = a_in @ wg.T, a_in @ wu.T
        s = torch.sigmoid(g)
        act = g * s * u
        out.index_add_(0, tok, wt[:, None] * (act @ wd.T))
        if d64 is None:
            return None
        z = d64[tok] @ wd
        dg = wt[:, None] * z * u * s * (1 + g * (1 - s))
        du = wt[:, None] * z * g * s
        if need_h:
            dh.index_add_(0, tok, dg @ wg + du @ wu)
        return (z * act).sum(1), dg, du, wt[:, None] * act

    for pool, name, n, base in ((0, "pub", E_pub, 0), (1, "priv", case["E_priv"], E_pub)):
        toks = torch.nonzero(allowed if pool else ~allowed).flatten()
        if toks.numel() == 0:
            continue
        r64 = w["router_" + name].double()
        z = h64[toks] @ r64.T
        top, sel = torch.sort(z, dim=1, descending=True, stable=True)
        top, sel = top[:, :k], sel[:, :k]
        prob = torch.softmax(z, dim=1)
        wt = torch.softmax(top, dim=1) if case["renorm"] else torch.gather(prob, 1, sel)
        idx[toks] = (sel + base).to(torch.int32)
        wts[toks] = wt
        gw = torch.zeros_like(wt)
        for e in range(n):
            row, rank = torch.nonzero(sel == e, as_tuple=True)
            if row.numel() == 0:
                continue
            tok = toks[row]
            r = expert(tok, wt[row, rank], w["gate_" + name][e].double(), w["up_" + name][e].double(),
                       w["down_" + name][e].double())
            if r is None:
                continue
            gw[row, rank] = r[0]
            if need_w and pool:
                grads["d_gate"][e] = r[1].T @ h64[tok]
                grads["d_up"][e] = r[2].T @ h64[tok]
                grads["d_down"][e] = d64[tok].T @ r[3]
        if d64 is None:
            continue
        s = (wt * gw).sum(1, keepdim=True)
        if case["renorm"]:
            dz = torch.zeros_like(z).scatter_(1, sel, wt * (gw - s))
        else:
            dz = -prob * s
            dz.scatter_add_(1, sel, wt * gw)
        if need_w and pool:
            grads["d_router"] = dz.T @ h64[toks]
        if need_h:
            dh.index_add_(0, toks, dz @ r64)
    one = torch.ones(T, dtype=torch.float64, device=h.device)
    every = torch.arange(T, device=h.device)
    for e in range(case["E_sh"]):
        expert(every, one, w["gate_sh"][e].double(), w["up_sh"][e].double(), w["down_sh"][e].double())
    return out, idx, wts, grads, dh


def exact(case, seed):
    mode = case["mode"]
    byte, cu = _requests(case, seed)
    policy = byte.repeat_interleave((cu[1:] - cu[:-1]).long()).cuda()
    h = _hidden(case, seed)
    if mode == "stack":
        x = h.double()
        for l in range(case["layers"]):
            x = x + _layer64(case, _inputs(case, seed, l), x, policy)[0]
        return x
    w = _inputs(case, seed)
    if mode in ("forward", "serve"):
        out, _, wts, _, _ = _layer64(case, w, h, policy)
        r = {"out": out, "idx": None, "w": wts}
        return dict(r, policy=None, audit=None) if mode == "serve" else r
    out, _, _, grads, dh = _layer64(case, w, h, policy, _dout(case, seed), need_w=mode != "input",
                                    need_h=mode != "private")
    if mode == "private":
        return {"out": out, "grads": grads}
    if mode == "input":
        return {"out": out, "d_hidden": dh}
    return {"out": out, "grads": grads, "d_hidden": dh}
