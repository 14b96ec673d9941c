"""Performance cases of the MoE-ViE layer library, through its Python binding of the C ABI.

A case is one call sequence a program makes on one MoE FFN layer:

  forward   moevie_moe_forward: inference on a batch of tokens
  train     moevie_moe_forward (keeping the selection), then moevie_moe_backward
  backward  moevie_moe_backward alone, on a selection of an earlier forward
  staged    the stages one by one: route, permute, expert FFN, shared expert, combine
  host      moevie_moe_forward_host: tokens from and to pinned host memory

Sizes are the repository's layer workloads (whole images or clips of 256 or 1024 patch
tokens) and ragged token counts between them.  Token counts 256 .. 65536, d 512 .. 1664,
8 .. 256 experts of width 100 .. 1024 (odd widths included), 1 .. 8 selected, GELU and
SwiGLU experts, with and without a shared expert, balanced and skewed expert loads.
"""
import math

import torch

from paper_2608_17402_gb300 import moevie


def _case(name, kind, T, d, E, k, h, hs=0, act="gelu", skew=0.0, hot=0, empty=0):
    c = {"kind": kind, "T": T, "d": d, "E": E, "k": k, "h": h, "hs": hs, "act": act,
         "skew": skew, "hot": hot, "empty": empty}
    return {"name": name, **c} if name else c


def listed():
    return [
        # One 224^2 image through the base model's layer: the smallest call, bound by latency
        # and launches.
        _case("base_1_image", "forward", 256, 768, 31, 3, 512, 512, "swiglu"),
        # Two images, few wide experts, no shared expert.
        _case("two_images", "forward", 512, 768, 16, 2, 768),
        # One 448^2 image at batch 1: every expert's weights are read for few rows each.
        _case("one_448_image", "forward", 1024, 1536, 64, 8, 768),
        # The ordinary inference batch: 32 images, 64 narrow experts and a shared expert twice
        # as wide.
        _case("images_32", "forward", 8192, 1024, 64, 8, 512, 1024),
        # The large model's layer, its width 684 no multiple of 8, on a ragged token count
        # (images of several sizes packed together).
        _case("large_ragged", "forward", 7003, 1024, 31, 3, 684, 684, "swiglu"),
        # The huge model's layer on eight 448^2 images: the most arithmetic per token.
        _case("huge_448", "forward", 8192, 1280, 31, 7, 854, 854, "swiglu"),
        # Four video clips of 32 frames: loads as trained routers give them on video, far from
        # balanced, some experts empty.
        _case("clips_4", "forward", 32768, 1536, 128, 8, 384, skew=0.55, empty=4),
        # The largest layer call: many narrow experts, one that every token selects.
        _case("stress", "forward", 65536, 1664, 256, 8, 416, skew=0.55, hot=1, empty=3),
        # A training step of the large model's layer: forward, then every gradient.
        _case("train_large", "train", 8192, 1024, 31, 3, 684, 684, "swiglu"),
        # The backward of the ordinary batch (activation checkpointing runs it apart).
        _case("backward_images_32", "backward", 8192, 1024, 64, 8, 512, 1024),
        # A program that drives the stages itself, on a ragged batch of about eight images.
        _case("staged_ragged", "staged", 2011, 1024, 64, 8, 512, 1024),
        # The video layer for a server whose tokens live in host memory.
        _case("host_clips_4", "host", 32768, 1536, 128, 8, 384, skew=0.55, empty=4),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges; no costlier than the largest listed one."""
    most = 0.7 * work(listed()[7])["flops"]
    while True:
        kind = rng.choice(["forward", "forward", "forward", "forward", "train", "backward", "staged", "host"])
        T = _log_uniform(rng, 256, 65536)
        if kind == "host":
            T = max(T, 2048)
        d = 8 * rng.randint(64, 208)
        E = _log_uniform(rng, 8, 256)
        k = rng.randint(1, min(8, E))
        h = _log_uniform(rng, 100, 1024)
        shared = rng.random() < 0.5 or kind == "staged"
        hs = (h if rng.random() < 0.6 else rng.randint(64, 1024)) if shared else 0
        act = "gelu" if kind == "staged" else rng.choice(["gelu", "swiglu"])
        skewed = rng.random() < 0.4 and E >= 16
        c = _case(None, kind, T, d, E, k, h, hs, act, 0.55 if skewed else 0.0,
                  1 if skewed and k > 1 and rng.random() < 0.5 else 0, rng.randint(0, 3) if skewed else 0)
        if work(c)["flops"] <= most:
            return c


def _offsets(c, rank):
    """Logit offsets of a skewed layer: a power law over the experts in the order `rank`
    (loads near Zipf's), hot experts that every token selects, and empty ones."""
    E, hot, empty = c["E"], c["hot"], c["empty"]
    o = -c["skew"] * torch.log(torch.arange(1, E + 1, dtype=torch.float64, device=rank.device))
    if hot:
        o[:hot] = 6.0
    if empty:
        o[E - empty:] = -12.0
    out = torch.empty_like(o)
    out[rank] = o
    return out.float()


def _tensors(c, seed):
    """The layer's inputs from the seed: tokens as after a LayerNorm, router weights of
    standard deviation 0.02, a small selection bias, expert weights of variance 1/fan_in."""
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    T, d, E, h, hs = c["T"], c["d"], c["E"], c["h"], c["hs"]

    def normal(shape, std=1.0):
        return (torch.randn(shape, generator=g, device="cuda") * std).to(torch.bfloat16)

    x = normal((T, d))
    W_r = torch.randn((d, E), generator=g, device="cuda") * 0.02
    b = torch.rand(E, generator=g, device="cuda") * 0.2 - 0.1
    t = {"x": x, "W_r": W_r, "b": b, "W1": normal((E, d, h), d ** -0.5), "W2": normal((E, h, d), h ** -0.5),
         "W3": None, "Ws1": None, "Ws2": None, "Ws3": None}
    if hs:
        t["Ws1"], t["Ws2"] = normal((d, hs), d ** -0.5), normal((hs, d), hs ** -0.5)
    if c["act"] == "swiglu":
        t["W3"] = normal((E, d, h), d ** -0.5)
        if hs:
            t["Ws3"] = normal((d, hs), d ** -0.5)
    if c["skew"]:
        rank = torch.randperm(E, generator=g, device="cuda")
        x[:, d - 1] = 1.0
        W_r[d - 1] = _offsets(c, rank)
    if c["kind"] in ("train", "backward"):
        t["dy"] = normal((T, d))
    return t


def prepare(case, seed):
    t = _tensors(case, seed)
    T, d, E, k, h, hs = (case[n] for n in ("T", "d", "E", "k", "h", "hs"))
    rows = {n: None if t[n] is None else moevie.moevie_pad_rows(t[n]) for n in ("W1", "W3", "Ws1", "Ws3")}
    s = {"kind": case["kind"], "k": k, "E": E, "x": t["x"],
         "layer": moevie.LayerWeights(W_r=t["W_r"], b=t["b"], W1=rows["W1"], W2=t["W2"], k=k, Ws1=rows["Ws1"],
                                      Ws2=t["Ws2"], lam=1.0, W3=rows["W3"], Ws3=rows["Ws3"])}
    chunks = moevie.host_chunks(T) if case["kind"] == "host" else 1
    if case["kind"] != "backward":
        s["ws"] = moevie.Workspace(-(-T // chunks), d, E, k, h, hs)
        s["y"] = torch.empty_like(t["x"])
    if case["kind"] in ("train", "backward"):
        s["dy"] = t["dy"]
        s["bws"] = moevie.BackwardWorkspace(T, d, E, k, h, hs, case["act"] == "swiglu")
    if case["kind"] == "backward":   # the selection the forward made
        s["idx"], _ = moevie.moevie_route(s["x"], t["W_r"], t["b"], k, moevie.Workspace(T, d, E, k, h, hs))
        torch.cuda.synchronize()
    if case["kind"] == "host":
        s["chunks"] = chunks
        s["x_host"] = torch.empty((T, d), dtype=torch.bfloat16, pin_memory=True)
        s["x_host"].copy_(t["x"])
        s["y_host"] = torch.empty((T, d), dtype=torch.bfloat16, pin_memory=True)
    return s


def run(state):
    s, kind, W = state, state["kind"], state["layer"]
    if kind == "forward":
        return moevie.moevie_moe_forward(W, s["x"], s["ws"], y=s["y"])
    if kind == "train":
        y, rt = moevie.moevie_moe_forward(W, s["x"], s["ws"], y=s["y"], routing=True)
        return {"y": y, "idx": rt["idx"], "counts": rt["counts"],
                **moevie.moevie_moe_backward(W, s["x"], s["dy"], rt["idx"], s["bws"])}
    if kind == "backward":
        return moevie.moevie_moe_backward(W, s["x"], s["dy"], s["idx"], s["bws"])
    if kind == "host":
        return moevie.moevie_moe_forward_host(W, s["x_host"], s["y_host"], s["x"], s["y"], s["ws"], s["chunks"])
    idx, gate = moevie.moevie_route(s["x"], W.W_r, W.b, s["k"], s["ws"])
    counts, offsets, perm, inv = moevie.moevie_permute(idx, s["E"], s["ws"])
    rows = moevie.moevie_expert_ffn(s["x"], perm, offsets, W.W1, W.W2, s["k"], s["ws"])
    shared = moevie.moevie_shared_expert(s["x"], W.Ws1, W.Ws2, s["ws"])
    y = moevie.moevie_combine(rows, inv, gate, s["k"], shared, W.lam, s["y"])
    return {"y": y, "idx": idx, "gate": gate, "counts": counts, "offsets": offsets, "perm": perm, "inv": inv}


def work(case):
    """Bytes: x, y, the router, the weights of the experts (those with rows) and the
    routing; for the backward also dy and every fp32 gradient.  Operations: the router's and
    the experts' products, for the backward those of the activations again, of dx and of the
    weights."""
    T, d, E, k, h, hs = (case[n] for n in ("T", "d", "E", "k", "h", "hs"))
    mats = 3 if case["act"] == "swiglu" else 2
    touched = min(E - case["empty"], T * k)
    weights = mats * d * (touched * h + hs)          # elements
    products = mats * d * (T * k * h + T * hs)       # multiply-adds of the experts
    fwd = {"bytes": 2 * 2 * T * d + 4 * d * E + 4 * E + 2 * weights + 8 * T * k,
           "flops": 2 * T * d * E + 2 * products}
    up = (mats - 1) * d * (T * k * h + T * hs)       # the up-projection again
    bwd = {"bytes": 2 * 2 * T * d + 4 * d * E + 2 * weights + 4 * T * k + 4 * T * d + 4 * d * E
                    + 4 * mats * d * (E * h + hs),
           "flops": 2 * T * k * d + 2 * up + 4 * products + 2 * T * k * d * 2}
    if case["kind"] == "backward":
        return bwd
    if case["kind"] == "train":
        return {n: fwd[n] + bwd[n] for n in fwd}
    return fwd


# ---------------------------------------------------------------- 64-bit results

def _act(c, u, v):
    return torch.nn.functional.silu(u) * v if c["act"] == "swiglu" else torch.nn.functional.gelu(u)


def _act_grad(c, u, v, da):
    """(du, dv) of the activation."""
    if c["act"] == "swiglu":
        sg = torch.sigmoid(u)
        return da * v * sg * (1 + u * (1 - sg)), da * u * sg
    phi = torch.exp(-0.5 * u * u) / math.sqrt(2 * math.pi)
    return da * (0.5 * (1 + torch.erf(u / math.sqrt(2))) + u * phi), None


def _route64(t, k):
    s = t["x"].double() @ t["W_r"].double()
    idx = torch.topk(torch.sigmoid(s) + t["b"].double(), k, dim=1).indices.sort(dim=1).values
    sg = torch.sigmoid(s.gather(1, idx))
    return idx, sg, sg / sg.sum(dim=1, keepdim=True)


def _ffn64(c, t, x, e):
    """(u, v, a, out) of expert e (None: the shared expert) on rows x."""
    w1, w2, w3 = ((t[n] if e is None else None if t[n] is None else t[n][e])
                  for n in (("Ws1", "Ws2", "Ws3") if e is None else ("W1", "W2", "W3")))
    u = x @ w1.double()
    v = x @ w3.double() if c["act"] == "swiglu" else None
    a = _act(c, u, v)
    return u, v, a, a @ w2.double()


def _forward64(c, t, idx, gate):
    x = t["x"].double()
    y = torch.zeros_like(x)
    for e in range(c["E"]):
        tok, j = (idx == e).nonzero(as_tuple=True)
        if tok.numel():
            y.index_add_(0, tok, gate[tok, j, None] * _ffn64(c, t, x[tok], e)[3])
    if c["hs"]:
        y += _ffn64(c, t, x, None)[3]
    return y


def _backward64(c, t, idx, sg, gate):
    x, dy = t["x"].double(), t["dy"].double()
    swiglu = c["act"] == "swiglu"
    g = {"dx": torch.zeros_like(x), "dW_r": None, "dW1": torch.zeros(t["W1"].shape, dtype=torch.float64, device="cuda"),
         "dW2": torch.zeros(t["W2"].shape, dtype=torch.float64, device="cuda")}
    if swiglu:
        g["dW3"] = torch.zeros_like(g["dW1"])
    dg = torch.zeros_like(gate)

    def expert(e, xe, dye, scale, w):
        u, v, a, out = _ffn64(c, t, xe, e)
        gdy = scale * dye
        du, dv = _act_grad(c, u, v, gdy @ w["W2"].double().T)
        dxe = du @ w["W1"].double().T
        if swiglu:
            dxe = dxe + dv @ w["W3"].double().T
        return dxe, xe.T @ du, a.T @ gdy, xe.T @ dv if swiglu else None, (dye * out).sum(dim=1)

    for e in range(c["E"]):
        tok, j = (idx == e).nonzero(as_tuple=True)
        if not tok.numel():
            continue
        w = {n: None if t[n] is None else t[n][e] for n in ("W1", "W2", "W3")}
        dxe, d1, d2, d3, dge = expert(e, x[tok], dy[tok], gate[tok, j, None], w)
        g["dx"].index_add_(0, tok, dxe)
        g["dW1"][e], g["dW2"][e] = d1, d2
        if swiglu:
            g["dW3"][e] = d3
        dg[tok, j] = dge
    ds = sg * (1 - sg) * (dg - (gate * dg).sum(dim=1, keepdim=True)) / sg.sum(dim=1, keepdim=True)
    dense = torch.zeros((c["T"], c["E"]), dtype=torch.float64, device="cuda").scatter_(1, idx, ds)
    g["dW_r"] = x.T @ dense
    g["dx"] += dense @ t["W_r"].double().T
    if c["hs"]:
        w = {"W1": t["Ws1"], "W2": t["Ws2"], "W3": t["Ws3"]}
        dxe, g["dWs1"], g["dWs2"], d3, _ = expert(None, x, dy, 1.0, w)
        g["dx"] += dxe
        if swiglu:
            g["dWs3"] = d3
    return g


def exact(case, seed):
    t = _tensors(case, seed)
    c, kind = case, case["kind"]
    idx, sg, gate = _route64(t, c["k"])
    if kind == "backward":
        return _backward64(c, t, idx, sg, gate)
    y = _forward64(c, t, idx, gate)
    if kind == "forward":
        return y
    if kind == "host":
        return y.cpu()
    flat = idx.reshape(-1)
    counts = torch.bincount(flat, minlength=c["E"])
    if kind == "train":
        return {"y": y, "idx": idx, "counts": counts, **_backward64(c, t, idx, sg, gate)}
    perm = torch.sort(flat, stable=True).indices
    inv = torch.empty_like(perm)
    inv[perm] = torch.arange(perm.numel(), device=perm.device)
    offsets = torch.nn.functional.pad(counts.cumsum(0), (1, 0))
    return {"y": y, "idx": idx, "gate": gate, "counts": counts, "offsets": offsets, "perm": perm, "inv": inv}
