"""Workloads whose speed matters to a program that serves a model with this library.

Every case goes through the public binding (paper_2605_10875_b200.binding), as a serving loop does: the packed
weights, the paged caches, the page tables and the workspace are there before the call, one call is one pass.
Shapes are those of the repository's workloads (synth.py): the tiny layer, the Llama-3.2-1B and the Llama-3.1-8B
layer, and a generic one with three query heads per kv-head; caches and hidden states are N(0, 1), weights
N(0, 0.02), norm gains 1 + N(0, 0.02), pages of 64 tokens in shuffled order, contexts uniform or lognormal,
actions mixed over the batch.  Calls that append write the same entry at the same place on every pass, so a state
can be run any number of times.
"""
import math
import statistics

import numpy as np
import torch

from paper_2605_10875_b200 import binding as sol

DEV = "cuda"
PAGE = 64
EPS = 1e-5
R_SET = (125, 250, 500, 1000)
P_SET = (0, 250, 500, 750)
B_SET = (4, 8, 16)
# Steps of several layers pass at 16 bits (12 and 16 where the quantizer sits on the MLP output) and keep every channel.
# Selections and codes amplify: a last-bit difference in one sum moves a code or swaps a channel at the threshold, the
# next layer's selections follow, and after 16 layers two correct programs are 7 % apart with pruned channels, 14 % with
# 4-bit rows, so their results could not be compared.  Single layers take every width and every prune rate.
B_SET_DEEP = (16,)
B_SET_OUTPUT = (12, 16)
MIX = -1                     # an action that differs from sequence to sequence

SHAPES = {
    "tiny": dict(d=256, hq=4, hkv=2, hd=64, ff=1024, theta=0.0),
    "generic": dict(d=768, hq=12, hkv=4, hd=64, ff=2080, theta=10000.0),
    "llama1b": dict(d=2048, hq=32, hkv=8, hd=64, ff=8192, theta=500000.0),
    "llama8b": dict(d=4096, hq=32, hkv=8, hd=128, ff=14336, theta=500000.0),
}


def _case(kind, shape="llama1b", layers=1, batch=1, context=0, sigma=0.0, r=MIX, p=MIX, b=MIX, quest=0, place=0, gate=0,
          tokens=0, name=None):
    c = dict(kind=kind, shape=shape, layers=layers, batch=batch, context=context, sigma=sigma, r=r, p=p, b=b, quest=quest,
             place=place, gate=gate, tokens=tokens)
    return dict(c, name=name) if name else c


def listed():
    return [
        # one small layer, everything in L2: the cost of a chain of dependent launches
        _case("layer", "tiny", 1, 4, 512, name="tiny_layer"),
        # one user's chat turn: a whole model step for a single sequence, bound by weights and latency
        _case("step", "llama1b", 16, 1, 1999, r=500, p=0, name="single_sequence_step"),
        # a layer of a small server, equal contexts
        _case("layer", "llama1b", 1, 16, 4096, b=16, name="layer_batch16"),
        # a model step at the batch and context of an offline run
        _case("step", "llama1b", 16, 32, 8192, p=0, name="step_batch32"),
        # a layer of the larger model: 128-wide heads, long contexts, dominated by cache reads
        _case("layer", "llama8b", 1, 64, 16384, name="layer_8b_batch64"),
        # a full server batch whose contexts differ by two orders of magnitude, one layer under every kind of action
        _case("layer", "llama1b", 1, 128, 4096, sigma=1.0, name="ragged_layer_batch128"),
        # the largest: the whole model step of that server
        _case("step", "llama1b", 16, 128, 4096, sigma=1.0, p=0, name="ragged_serving_step"),
        # the step as called by a server that keeps its tokens and actions on the host
        _case("host_step", "llama1b", 16, 24, 2048, sigma=0.7, p=0, name="host_step_batch24"),
        # the paper's own forms of the three knobs: page selection per query head, input gating, output quantizer
        _case("layer", "llama1b", 1, 96, 4096, sigma=1.0, quest=16, place=1, gate=1, name="quest_layer_batch96"),
        # the periodic dense pass over a horizon's last 16 tokens
        _case("refresh", "llama1b", 4, 32, 4096, sigma=1.0, r=1000, p=0, b=16, tokens=16, name="refresh_16_tokens"),
        # the attention alone inside someone else's layer, odd batch, 128-wide heads
        _case("attention", "llama8b", 1, 31, 5000, sigma=0.8, name="attention_ragged_hd128"),
        # the pruned MLP alone at a batch where pruned rows of the down projection are really not read
        _case("mlp", "llama8b", 1, 3, p=500, name="mlp_batch3"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "layer", "layer", "host_step", "quest", "quest", "refresh", "attention",
                       "mlp", "quant"])
    shape = rng.choice(["tiny", "generic", "llama1b", "llama1b", "llama1b", "llama8b"])
    S = SHAPES[shape]
    if kind == "quant":
        return _case("quant", shape, 1, _log(rng, 1, 4096))
    if kind == "mlp":
        return _case("mlp", shape, 1, _log(rng, 1, 128), p=rng.choice([MIX, 0, 250, 500, 750]))
    layers = 1 if kind in ("layer", "attention") else rng.randint(1, 4 if kind in ("quest", "refresh") else {"llama8b": 6}.get(shape, 16))
    batch = _log(rng, 1, 48 if kind == "refresh" else 128)
    context = _log(rng, 64, 24000)
    sigma = rng.choice([0.0, 0.5, 1.0])
    room = 8e9 / (layers * batch * S["hkv"] * S["hd"] * 4 * math.exp(sigma * sigma / 2))  # at most 8 GB of cache
    context = max(33, min(context, int(room)))
    c = _case(kind, shape, layers, batch, context, sigma, rng.choice([MIX, MIX, 125, 250, 500, 1000]),
              rng.choice([MIX, MIX, 0, 500]), rng.choice([MIX, MIX, 4, 8, 16]) if layers == 1 else MIX)
    if layers > 1:  # see B_SET_DEEP; of a short context's few kept tokens each one counts as much as a channel
        c.update(p=0, r=c["r"] if context >= 1500 else 1000)
    if kind == "quest":
        c.update(kind="step", quest=rng.choice([4, 8, 16, 16, 32, 64]), place=rng.randint(0, 1), gate=rng.randint(0, 1), b=MIX)
    if kind == "refresh":
        c.update(tokens=rng.choice([4, 8, 16, 16, 16]), r=1000, p=0, b=16)
    if kind == "attention":
        c.update(p=MIX, b=MIX, quest=rng.choice([0, 0, 0, 16]))
    return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
_NAMES = ("w_qkv", "w_o", "w_gate", "w_up", "w_down", "gamma1", "gamma2", "k", "v", "h", "q", "x")


def _normal(seed, name, layer, shape, mean=0.0, std=1.0):
    g = torch.Generator(device=DEV)
    g.manual_seed((int(seed) * 1000003 + _NAMES.index(name)) * 1009 + layer)
    return torch.empty(shape, dtype=torch.bfloat16, device=DEV).normal_(mean, std, generator=g)


def _weights(c, seed, layer):
    S = SHAPES[c["shape"]]
    d, ff, qo, n = S["d"], S["ff"], S["hq"] * S["hd"], (S["hq"] + 2 * S["hkv"]) * S["hd"]
    w = dict(w_qkv=(n, d), w_o=(d, qo), w_gate=(ff, d), w_up=(ff, d), w_down=(ff, d))
    if c["kind"] == "mlp":
        w = {k: w[k] for k in ("w_gate", "w_up", "w_down")}
    out = {k: _normal(seed, k, layer, s, 0.0, 0.02) for k, s in w.items()}
    if c["kind"] != "mlp":
        out.update({k: _normal(seed, k, layer, (d,), 1.0, 0.02) for k in ("gamma1", "gamma2")})
    return out


def _lengths(c):
    """Context lengths of the batch: the middles of B equal shares of the distribution, shortest first."""
    B, T = c["batch"], c["context"]
    if not c["sigma"]:
        return [T] * B
    z = [statistics.NormalDist().inv_cdf((i + 0.5) / B) for i in range(B)]
    return [max(min(T, 256), min(32768, int(round(T * math.exp(c["sigma"] * x))))) for x in z]


def _plan(c, seed):
    """Lengths, actions and page table of a batch, on the host."""
    rng = np.random.default_rng([int(seed), 77])
    B = c["batch"]
    bits = B_SET_OUTPUT if c["place"] else B_SET if c["layers"] == 1 else B_SET_DEEP

    def action(v, values):
        return rng.permutation(np.resize(np.asarray(values, np.int32), B)) if v == MIX else np.full(B, v, np.int32)

    lens = rng.permutation(np.asarray(_lengths(c), np.int32)) if c["context"] else np.zeros(B, np.int32)
    pages = -(-lens // PAGE)
    ids = rng.permutation(int(pages.sum())).astype(np.int32)
    table = np.zeros((B, max(1, int(pages.max()))), np.int32)
    at = 0
    for i, n in enumerate(pages):
        table[i, :n] = ids[at:at + n]
        at += n
    return dict(lens=lens, table=table, pages=at, r=action(c["r"], R_SET), p=action(c["p"], P_SET), b=action(c["b"], bits))


def _pools(c, seed, layer, pages):
    S = SHAPES[c["shape"]]
    shape = (pages, S["hkv"], PAGE, S["hd"])
    return _normal(seed, "k", layer, shape), _normal(seed, "v", layer, shape)


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.int32)).to(DEV)


def _shape(c):
    S = SHAPES[c["shape"]]
    return sol.make_shape(S["d"], S["hq"], S["hkv"], S["hd"], S["ff"], PAGE, EPS, S["theta"], 0, 1,
                          quant_placement=c["place"], mlp_prune=c["gate"],
                          token_select=sol.SELECT_QUEST_PAGES if c["quest"] else sol.SELECT_TOKENS, quest_page_size=c["quest"])


def _pack(shape, kind, a, b=None):
    n = sol.packed_weight_bytes(shape, kind)
    out = torch.empty(n, dtype=torch.uint8, device=DEV)
    sol.pack_weights(shape, kind, a, b, out, n)
    return out


def _workspace(st, rows, pages):
    st["ws_bytes"] = sol.workspace_bytes(st["shape"], rows, pages)
    st["ws"] = torch.empty(st["ws_bytes"], dtype=torch.uint8, device=DEV)
    sol.workspace_init(st["ws"], st["ws_bytes"])


def prepare(case, seed):
    c, S, B = case, SHAPES[case["shape"]], case["batch"]
    plan = _plan(c, seed)
    st = dict(kind=c["kind"], B=B, shape=_shape(c))
    for k in ("r", "p", "b"):
        st[k] = _dev(plan[k])
    if c["kind"] == "quant":
        st["x"] = _normal(seed, "x", 0, (B, S["d"]))
        st["codes"] = torch.zeros((B, S["d"]), dtype=torch.int8, device=DEV)
        st["scales"] = torch.zeros(B, dtype=torch.float32, device=DEV)
        st["xhat"] = torch.zeros((B, S["d"]), dtype=torch.bfloat16, device=DEV)
        return st
    if c["kind"] == "mlp":
        w = _weights(c, seed, 0)
        st["w"] = (_pack(st["shape"], sol.W_GATE_UP, w["w_gate"], w["w_up"]), _pack(st["shape"], sol.W_DOWN, w["w_down"]))
        st["x"] = _normal(seed, "x", 0, (B, S["d"]))
        st["out"] = torch.zeros((B, S["d"]), dtype=torch.bfloat16, device=DEV)
        _workspace(st, B, 1)
        return st
    table, lens = _dev(plan["table"]), _dev(plan["lens"])
    max_pages = plan["table"].shape[1]
    st["pools"], st["metas"], st["kvs"], st["layers"], st["keep"] = [], [], [], [], [table, lens]
    for layer in range(c["layers"]):
        k, v = _pools(c, seed, layer, plan["pages"])
        meta = None
        if c["quest"]:
            meta = torch.zeros(sol.quest_meta_bytes(st["shape"], plan["pages"]) // 2, dtype=torch.bfloat16, device=DEV)
            st["metas"].append(meta)
        kv = sol.make_kv(k, v, table, lens, max_pages, plan["pages"], meta)
        if c["quest"]:  # the extrema that a prefill leaves behind
            sol.quest_build_meta(st["shape"], kv, B)
        st["pools"] += [k, v]
        st["kvs"].append(kv)
        if c["kind"] != "attention":
            w = _weights(c, seed, layer)
            packed = [_pack(st["shape"], sol.W_QKV, w["w_qkv"]), _pack(st["shape"], sol.W_O, w["w_o"]),
                      _pack(st["shape"], sol.W_GATE_UP, w["w_gate"], w["w_up"]), _pack(st["shape"], sol.W_DOWN, w["w_down"]),
                      w["gamma1"], w["gamma2"]]
            st["layers"].append(sol.make_weights(*packed))
            st["keep"] += packed
    if c["kind"] == "attention":
        st["q"] = _normal(seed, "q", 0, (B, S["hq"], S["hd"]))
        st["out"] = torch.zeros_like(st["q"])
    elif c["kind"] == "refresh":
        st["tokens"] = min(c["tokens"], int(plan["lens"].min()))
        st["h"] = _normal(seed, "h", 0, (B, st["tokens"], S["d"]))
        st["out"] = torch.zeros_like(st["h"])
    else:
        st["h"] = _normal(seed, "h", 0, (B, S["d"]))
        st["out"] = torch.zeros_like(st["h"])
    if c["kind"] == "host_step":
        st["h"] = st["h"].cpu().pin_memory()
        st["out"] = st["out"].cpu().pin_memory()
        for k in ("r", "p", "b"):
            st[k] = torch.from_numpy(plan[k]).pin_memory()
        st["lens"] = torch.from_numpy(plan["lens"]).pin_memory()
    rows = min(B, 128 // st["tokens"]) * st["tokens"] if c["kind"] == "refresh" else B
    _workspace(st, rows, max_pages)
    return st


def run(state):
    st = state
    kind, shape, B = st["kind"], st["shape"], st["B"]
    stream = torch.cuda.current_stream()
    if kind == "quant":
        sol.quant_act(st["x"], B, st["x"].shape[1], st["b"], st["codes"], st["scales"], st["xhat"], stream=stream)
        return {"codes": st["codes"], "scales": st["scales"], "xhat": st["xhat"]}
    if kind == "mlp":
        sol.pruned_swiglu_mlp(shape, st["x"], st["w"][0], st["w"][1], B, st["p"], st["out"], None, None, st["ws"],
                              st["ws_bytes"], stream=stream)
        return {"out": st["out"]}
    if kind == "attention":
        sol.sparse_decode_attn(shape, st["q"], st["kvs"][0], B, st["r"], st["out"], None, None, st["ws"], st["ws_bytes"],
                               stream=stream)
        return {"out": st["out"]}
    if kind == "layer":
        sol.decode_layer(shape, st["layers"][0], st["kvs"][0], B, st["h"], st["out"], st["r"], st["p"], st["b"], None,
                         st["ws"], st["ws_bytes"], stream=stream)
    elif kind == "step":
        sol.decode_step(shape, st["layers"], st["kvs"], B, st["h"], st["out"], None, st["r"], st["p"], st["b"], st["ws"],
                        st["ws_bytes"], stream=stream)
    elif kind == "host_step":
        sol.decode_step_host(shape, st["layers"], st["kvs"], B, st["h"], st["out"], st["r"], st["p"], st["b"], st["lens"],
                             st["ws"], st["ws_bytes"], stream=stream)
    else:
        sol.kv_refresh(shape, st["layers"], st["kvs"], B, st["tokens"], st["h"], st["out"], st["ws"], st["ws_bytes"],
                       stream=stream)
    return {"out": st["out"], "pools": st["pools"], "extrema": st["metas"]}


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def work(case):
    c, S, B = case, SHAPES[case["shape"]], case["batch"]
    d, ff, hq, hkv, hd = S["d"], S["ff"], S["hq"], S["hkv"], S["hd"]
    if c["kind"] == "quant":
        return {"bytes": B * d * 5 + 8 * B, "flops": 3 * B * d}
    values = np.resize(np.asarray(P_SET), B) if c["p"] == MIX else np.full(B, c["p"])
    dense = c["kind"] == "refresh" or c["gate"]
    union = 1.0 if dense else 1.0 - float(np.prod(np.sort(values / 1000.0)))  # rows of W_down that some token keeps
    kept = 1.0 if dense else 1.0 - float(values.mean()) / 1000.0
    mlp_bytes, mlp_flops = 2 * d * ff * (2 + union), 2 * d * ff * (2 + kept)  # a layer's, and a token's
    if c["kind"] == "mlp":
        return {"bytes": mlp_bytes + 4 * B * d, "flops": B * mlp_flops}
    total = sum(_lengths(c))
    rates = np.resize(np.asarray(R_SET), B) if c["r"] == MIX else np.full(B, c["r"])
    r = 1.0 if c["kind"] == "refresh" else float(rates.mean()) / 1000.0
    row = 2 * hkv * hd  # bytes of one token's keys, or of its values
    if c["quest"] and c["kind"] != "refresh":  # extrema, then both rows of what some head of a kv-head keeps
        some = 1.0 - float(np.mean((1.0 - rates / 1000.0) ** (hq // hkv)))
        attn_bytes = total * row * (2.0 / c["quest"] + 2 * some)
        attn_flops = 2 * total * hq * hd * (2.0 / c["quest"] + 2 * r)
    else:
        attn_bytes = total * row * (1 + r)
        attn_flops = 2 * total * hq * hd * (1 + r)
    if c["kind"] == "attention":
        return {"bytes": attn_bytes + 4 * B * hq * hd, "flops": attn_flops}
    n = c["tokens"] if c["kind"] == "refresh" else 1
    proj = d * hd * (2 * hq + 2 * hkv)
    bytes_ = c["layers"] * (2 * proj + mlp_bytes + attn_bytes + 2 * B * n * row) + 4 * B * n * d
    return {"bytes": bytes_, "flops": c["layers"] * (B * n * (2 * proj + mlp_flops) + n * attn_flops)}


def tolerance(case):
    if case["kind"] == "quant":
        return "exact"
    # Measured against exact(): 1.7e-3 (the rounding of the output to 16 bits) for the attention, the MLP and dense
    # passes; up to 1.3e-2 where a code of 4 bits or a selection falls the other way on a last-bit difference.
    return {"rel": 7e-3 if case["kind"] in ("attention", "mlp", "refresh") else 3e-2}


# ---------------------------------------------------------------------------
# the same results in 64 bits, with plain torch
# ---------------------------------------------------------------------------
def _quantize(x, bits, passthrough):
    """Rows of float32 values as the quantizer returns them (codes decided in float32, as the method defines them);
    from 16 bits on what `passthrough` makes of the row."""
    q = torch.pow(2.0, (bits - 1).double()).float() - 1
    q = torch.where(bits >= 16, torch.ones_like(q), q)[:, None]
    a = x.abs().amax(dim=1, keepdim=True)
    s = a / q
    codes = torch.where(s > 0, torch.round(x / s), torch.zeros_like(x)).clamp(-q, q)
    wide = (bits >= 16)[:, None]
    return (torch.where(wide, torch.zeros_like(codes), codes), torch.where(wide, torch.ones_like(s), s)[:, 0],
            torch.where(wide, passthrough(x), codes.double() * s.double()))


def _top(score, k):
    """Mask of the k largest entries of each row (ties: lower index)."""
    order = torch.argsort(score, dim=-1, descending=True, stable=True)[..., :k]
    return torch.zeros(score.shape, dtype=torch.bool, device=score.device).scatter_(-1, order, True)


def _mlp(x, w, p, ff):
    t = x @ w["w_gate"].double().T
    t = t / (1 + torch.exp(-t)) * (x @ w["w_up"].double().T)
    kept = [((1000 - int(pi)) * ff + 999) // 1000 for pi in p]
    for i, m in enumerate(kept):
        if m < ff:
            t[i] = torch.where(_top(t[i].abs(), m), t[i], torch.zeros_like(t[i]))
    return t @ w["w_down"].double()


def _norm(h, gamma):
    return h * gamma.double() / torch.sqrt((h * h).mean(-1, keepdim=True) + EPS)


def _rotate(v, pos, theta):
    if not theta:
        return v
    hd = v.shape[-1]
    ang = pos[:, None].double() * torch.pow(torch.tensor(theta, dtype=torch.float64, device=DEV),
                                            -2.0 * torch.arange(hd // 2, dtype=torch.float64, device=DEV) / hd)
    cos, sin = ang.cos()[:, None], ang.sin()[:, None]
    lo, hi = v[..., :hd // 2], v[..., hd // 2:]
    return torch.cat([lo * cos - hi * sin, hi * cos + lo * sin], -1)


def _attend(c, q, k_pool, v_pool, plan, n):
    """q [B * n][hq][hd], the n newest tokens of every sequence; one of them takes part in a selection."""
    S = SHAPES[c["shape"]]
    hq, hkv, hd = S["hq"], S["hkv"], S["hd"]
    G, out = hq // hkv, torch.zeros_like(q)
    for i, T in enumerate(plan["lens"].tolist()):
        pages = torch.from_numpy(plan["table"][i, :-(-T // PAGE)].astype(np.int64)).to(DEV)
        K = k_pool[pages].transpose(0, 1).reshape(hkv, -1, hd)[:, :T].double()
        V = v_pool[pages].transpose(0, 1).reshape(hkv, -1, hd)[:, :T].double()
        rows = q[i * n:(i + 1) * n].reshape(n, hkv, G, hd).permute(1, 2, 0, 3).reshape(hkv, G * n, hd)
        dots = rows @ K.transpose(1, 2)  # [hkv][G * n][T]
        if c["kind"] == "refresh":
            late = torch.arange(T, device=DEV)[None] > torch.arange(T - n, T, device=DEV)[:, None]
            dots = dots.masked_fill(late.repeat(G, 1)[None], -math.inf)
        elif c["quest"]:
            P = -(-T // c["quest"])
            pad = P * c["quest"] - T
            top = torch.nn.functional.pad(K, (0, 0, 0, pad), value=-math.inf).view(hkv, P, c["quest"], hd).amax(2)
            low = torch.nn.functional.pad(K, (0, 0, 0, pad), value=math.inf).view(hkv, P, c["quest"], hd).amin(2)
            score = rows.clamp(min=0) @ top.transpose(1, 2) + rows.clamp(max=0) @ low.transpose(1, 2)
            score[..., -1] = math.inf  # the newest token's page is always kept
            budget = max(1, min(P, -(-((int(plan["r"][i]) * T + 999) // 1000) // c["quest"])))
            keep = _top(score, budget).repeat_interleave(c["quest"], dim=-1)[..., :T]
            dots = dots.masked_fill(~keep, -math.inf)
        else:
            score = dots.sum(1)
            score[..., -1] = math.inf  # the newest token is always kept
            keep = _top(score, max(1, min(T, (int(plan["r"][i]) * T + 999) // 1000)))
            dots = dots.masked_fill(~keep[:, None], -math.inf)
        o = torch.softmax(dots / math.sqrt(hd), -1) @ V
        out[i * n:(i + 1) * n] = o.reshape(hkv, G, n, hd).permute(2, 0, 1, 3).reshape(n, hq, hd)
    return out


def exact(case, seed):
    c, S, B = case, SHAPES[case["shape"]], case["batch"]
    hq, hkv, hd, ff = S["hq"], S["hkv"], S["hd"], S["ff"]
    plan = _plan(c, seed)
    bf16 = lambda x: x.bfloat16().double()  # noqa: E731
    if c["kind"] == "quant":
        x = _normal(seed, "x", 0, (B, S["d"]))
        codes, scales, _ = _quantize(x.float(), _dev(plan["b"]), lambda v: v.double())
        operand = torch.where((_dev(plan["b"]) >= 16)[:, None], x.double(), codes.double())
        return {"codes": codes.to(torch.int8), "scales": scales.double(), "xhat": operand}
    if c["kind"] == "mlp":
        return {"out": _mlp(_normal(seed, "x", 0, (B, S["d"])).double(), _weights(c, seed, 0), plan["p"], ff)}
    if c["kind"] == "attention":
        k, v = _pools(c, seed, 0, plan["pages"])
        return {"out": _attend(c, _normal(seed, "q", 0, (B, hq, hd)).double(), k, v, plan, 1)}
    n = 1
    if c["kind"] == "refresh":
        n = min(c["tokens"], int(plan["lens"].min()))
        plan.update(p=np.zeros(B * n, np.int32), b=np.full(B * n, 16, np.int32))
    bits = _dev(plan["b"])
    in_bits = torch.full_like(bits, 16) if c["place"] else bits
    pos = (plan["lens"][:, None] - n + np.arange(n)[None]).reshape(-1)  # of every row, n rows per sequence
    row_seq = np.repeat(np.arange(B), n)
    page = torch.from_numpy(plan["table"][row_seq, pos // PAGE].astype(np.int64)).to(DEV)
    slot = torch.from_numpy((pos % PAGE).astype(np.int64)).to(DEV)
    pos = torch.from_numpy(pos.astype(np.int64)).to(DEV)
    h = _normal(seed, "h", 0, (B, n, S["d"]) if c["kind"] == "refresh" else (B, S["d"])).reshape(B * n, S["d"]).double()
    for layer in range(c["layers"]):
        w = _weights(c, seed, layer)
        k_pool, v_pool = _pools(c, seed, layer, plan["pages"])
        x = _quantize(_norm(h, w["gamma1"]).float(), in_bits, bf16)[2]
        qkv = (x @ w["w_qkv"].double().T).view(B * n, hq + 2 * hkv, hd)
        q, k = _rotate(qkv[:, :hq], pos, S["theta"]), _rotate(qkv[:, hq:hq + hkv], pos, S["theta"])
        k_pool[page, :, slot] = k.bfloat16()
        v_pool[page, :, slot] = qkv[:, hq + hkv:].bfloat16()
        a = _attend(c, q, k_pool, v_pool, plan, n)
        h = h + a.reshape(B * n, hq * hd) @ w["w_o"].double().T
        x32 = _norm(h, w["gamma2"]).float()
        p = plan["p"]
        if c["gate"]:
            for i in range(B * n):
                x32[i] *= _top(x32[i].abs(), ((1000 - int(p[i])) * S["d"] + 999) // 1000)
            p = np.zeros(B * n, np.int32)
        z = _mlp(_quantize(x32, in_bits, bf16)[2], w, p, ff)
        if c["place"]:
            z = torch.where((bits >= 16)[:, None], z, _quantize(z.float(), bits, bf16)[2])
        h = h + z
    out = h.view(B, n, S["d"]) if c["kind"] == "refresh" else h
    # caches and extrema: one entry per sequence and layer is new, rounded to 16 bits, the rest is input
    return {"out": out, "pools": [None] * (2 * c["layers"]), "extrema": [None] * (c["layers"] if c["quest"] else 0)}
