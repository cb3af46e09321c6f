"""Work that users of this package have it do, as cases of one pass each through the public entry points.

A case is a routed prefill layer (``RoutedPrefillLayer.forward``: probe, candidate evaluation, routing, index lists,
attention, certificate in one call), the same layer replayed from a CUDA graph, the same layer fed by its producer
(``forward_from_hidden``), or the package's dense causal attention.  Inputs are drawn on the GPU from the seed.
"""
import math
import random

import torch

import paper_2608_29058_b200 as rs

D = 128

# Candidate libraries: the online default (None), the single vertical-slash budget of the 4K one-head workload, the four
# fixed patterns of the 32K fixed-route workload, and a small one for short prompts.
LIBRARIES = {
    "online": None,
    "one_head": [(rs.RS_VERTICAL_SLASH, 256, 512), (rs.RS_DENSE, 0, 0)],
    "fixed": [(rs.RS_A_SHAPE, 128, 1024), (rs.RS_VERTICAL_SLASH, 1000, 6096), (rs.RS_BLOCK_SPARSE, 100, 0), (rs.RS_DENSE, 0, 0)],
    "small": [(rs.RS_A_SHAPE, 8, 128), (rs.RS_VERTICAL_SLASH, 32, 48), (rs.RS_BLOCK_SPARSE, 3, 0), (rs.RS_DENSE, 0, 0)],
}


def _layer(name, n, hq, hkv, segments=1, library="online", recipe="archetype", routes="online", mixture=False,
           out="bf16", budget=0.15, cert=0.05, kind="layer"):
    return {"name": name, "kind": kind, "n": n, "hq": hq, "hkv": hkv, "segments": segments, "library": library,
            "recipe": recipe, "routes": routes, "mixture": mixture, "out": out, "budget": budget, "cert": cert}


def listed():
    return [
        # A short prompt on a small layer: the smallest call, launches and latency.
        _layer("layer_1k", 1024, 4, 2, library="small", recipe="planted", out="fp32", budget=0.4, cert=0.8),
        # One head at 4K (the repository's first workload), call by call.
        _layer("layer_4k_1head", 4096, 1, 1, library="one_head", recipe="planted", budget=0.6, cert=-1.0),
        # The same from a captured graph, new inputs copied in: how a server runs launch-bound sizes.
        _layer("graph_4k_1head", 4096, 1, 1, library="one_head", recipe="planted", budget=0.6, cert=-1.0, kind="graph"),
        # An 8B-shaped layer on a prompt whose length is 125 blocks: no multiple of the 128-row tile.
        _layer("layer_8k_odd", 8000, 32, 8),
        # The same layer at 16K: attention and the stages around it both count.
        _layer("layer_16k", 16384, 32, 8),
        # 32K with routes fixed ahead of time, all four patterns in one launch.
        _layer("layer_32k_fixed", 32768, 32, 8, library="fixed", recipe="planted", routes="fixed", budget=1.0, cert=-1.0),
        # Routing that looks at the whole query mixture (uncertainty and line lists), an odd length, fp32 output.
        _layer("layer_40k_mixture", 40000, 32, 8, mixture=True, out="fp32"),
        # The long-context layer the framework is built for.
        _layer("layer_128k", 131072, 32, 8),
        # Long context with four segments of different structure, each routed on its own.
        _layer("layer_128k_segments", 131072, 32, 8, segments=4, recipe="segments"),
        # Dense causal attention: a short batch-one prompt, and the audit of a 32K layer.
        {"name": "dense_4k", "kind": "dense", "n": 4096, "hq": 32, "hkv": 8, "segments": 1, "recipe": "planted", "out": "bf16"},
        {"name": "dense_32k", "kind": "dense", "n": 32768, "hq": 32, "hkv": 8, "segments": 1, "recipe": "archetype", "out": "bf16"},
        # From hidden states: QKV projection with rotary embedding, then the layer on what it wrote.
        {"name": "hidden_16k", "kind": "hidden", "n": 16384, "hq": 32, "hkv": 8, "segments": 1, "d_model": 4096},
    ]


def _blocks(rng, lo, hi):
    """A length between lo and hi (tokens), spread over the logarithm, a multiple of 64 and as often odd as even in blocks."""
    return 64 * max(1, round(math.exp(rng.uniform(math.log(lo), math.log(hi))) / 64))


def _windows_fit(bounds):
    """Candidate evaluation refuses a segment end just behind an A-shape window (sink and window would overlap there)."""
    return not any(w < q1 < w + 192 for q1 in bounds[1:] for w in (1024, 2048, 4096, 8192))


def draw(rng):
    while True:
        case = _draw(rng)
        if case.get("library") in ("fixed", "small", "one_head") or case["kind"] == "dense" or _windows_fit(_bounds(case["n"], case["segments"])):
            case.pop("name", None)
            if all(any(k != "name" and x[k] != case.get(k) for k in x) for x in listed()):
                return case


def _draw(rng):
    kind = rng.choices(["layer", "fixed", "small", "graph", "dense", "hidden"], [6, 2, 2, 1, 3, 1])[0]
    hq, hkv = rng.choice([(8, 2), (16, 4), (32, 8), (32, 8)])
    if kind == "small":
        return _layer("", _blocks(rng, 1024, 8192), 4, rng.choice([1, 2, 4]), library="small", recipe="planted",
                      out=rng.choice(["bf16", "fp32"]), budget=0.4, cert=0.8)
    if kind == "graph":
        return _layer("", _blocks(rng, 1024, 8192), 1, 1, library="one_head", recipe="planted", budget=0.6, cert=-1.0, kind="graph")
    if kind == "dense":
        return {"kind": "dense", "n": _blocks(rng, 1024, 40960), "hq": hq, "hkv": hkv, "segments": rng.choice([1, 1, 3]),
                "recipe": "planted", "out": rng.choice(["bf16", "bf16", "fp32"])}
    if kind == "hidden":
        return {"kind": "hidden", "n": _blocks(rng, 1024, 24576), "hq": 32, "hkv": 8, "segments": 1, "d_model": rng.choice([2048, 4096])}
    if kind == "fixed":
        return _layer("", _blocks(rng, 4096, 65536), hq, hkv, library="fixed", recipe="planted", routes="fixed", budget=1.0, cert=-1.0)
    n, segments = _blocks(rng, 4096, 131072), rng.choice([1, 1, 1, 2, 4])
    if segments > 1 and n < 16384:
        segments = 1
    return _layer("", n, hq, hkv, segments=segments, recipe="segments" if segments > 1 else "archetype",
                  mixture=n <= 65536 and rng.random() < 0.25, out=rng.choice(["bf16", "bf16", "fp32"]))


def _bounds(n, segments):
    return [64 * ((n // 64) * s // segments) for s in range(segments + 1)]


# ------------------------------------------------------------------------------------------------------- inputs
def _unit(gen, lo):
    """A random direction outside the first `lo` dimensions (those carry the rotary-like term)."""
    u = torch.randn(D, generator=gen, device="cuda")
    u[:lo] = 0.0
    return u / u.norm()


def _relative(n, pairs, boost, short, long):
    """[n, 2 pairs] rows c (cos, sin)(2 pi p / P_f): a contribution to Q.K that depends on i - j only."""
    c = math.sqrt(boost * math.sqrt(D) / pairs)
    periods = torch.logspace(math.log10(short), math.log10(long), pairs, device="cuda", dtype=torch.float64)
    ang = 2.0 * math.pi * torch.arange(n, device="cuda", dtype=torch.float64)[:, None] / periods[None, :]
    return torch.stack([c * torch.cos(ang), c * torch.sin(ang)], dim=2).reshape(n, 2 * pairs).float()


def _planted(case, gen, r):
    """Sinks on keys 0..3, eight vertical keys, local bias; constants that do not grow with the length."""
    n, hq, hkv = case["n"], case["hq"], case["hkv"]
    Q, K, V = (torch.empty((h, n, D), dtype=torch.bfloat16, device="cuda") for h in (hq, hkv, hkv))
    table = _relative(n, 8, 6.0, 512.0, 8.0 * n)
    for g in range(hkv):
        u, kr = _unit(gen, 0), torch.randn((n, D), generator=gen, device="cuda")
        boost = torch.zeros(n, device="cuda")
        boost[torch.tensor(r.sample(range(4, n - 64), 8), device="cuda")] = r.uniform(1.5, 4.5)
        boost[:4] = r.uniform(2.0, 6.0)
        k = kr + 4.0 * boost[:, None] * u
        k[:, :16] += table
        K[g] = k
        V[g] = torch.randn((n, D), generator=gen, device="cuda")
        for h in range(g * (hq // hkv), (g + 1) * (hq // hkv)):
            q = torch.randn((n, D), generator=gen, device="cuda") + r.uniform(2.0, 6.0) * u + r.uniform(0.25, 0.75) * kr
            q[:, :16] += table
            Q[h] = q
    return Q, K, V


def _archetypes(case, gen, r):
    """Heads of four kinds dealt to every KV group: local with sinks, vertical keys, separated blocks of the query's
    topic, and diffuse; strengths grow with log(n) so that structure keeps its share of the mass at every length.  With
    recipe "segments" the structure also switches from segment to segment: local text, a delimiter key every 257
    tokens, 16 needle keys copied to 8 places each, no structure at all."""
    n, hq, hkv = case["n"], case["hq"], case["hkv"]
    group, sd, grow, top, resp = hq // hkv, math.sqrt(D), math.log(max(n, 4096) / 4096.0), 14.5, 4.0
    pairs = 28
    lo = 2 * pairs
    drop = {"local": (0.5, 6.0, 0.0, None), "vertical": (0.5, 0.0, 0.5, None), "topic": (2.0, 6.0, 1.0, 0.0), "diffuse": (7.0, 8.0, 7.0, None)}
    jit = lambda a=0.25: r.uniform(-a, a)
    bounds, switched = _bounds(n, case["segments"]), case["recipe"] == "segments"
    order = r.sample(["local", "delimiter", "needle", "diffuse"], 4)
    kinds = [order[s % 4] if switched else "planted" for s in range(case["segments"])]
    heads = []
    for g in range(hkv):
        deal = ["local", "vertical", "topic", "local" if g % 2 == 0 else "vertical"][:group]
        if g % 3 == 2:
            deal[-1] = "diffuse"
        heads += [(k, 0.5 if k == "diffuse" else r.uniform(0.1, 0.3)) for k in r.sample(deal, len(deal))]
    boosts = [top - drop[k][2] - lam * sd - 0.7 + grow + jit() for k, lam in heads]
    mean_boost = sum(boosts) / len(boosts)
    table = _relative(n, pairs, mean_boost, 37.0, 5300.0)
    amp, gain = torch.ones(n, 1, device="cuda"), torch.ones(n, 1, device="cuda")
    for a, b, k in zip(bounds[:-1], bounds[1:], kinds):
        amp[a:b] = {"local": math.sqrt(8.0 / mean_boost), "diffuse": 0.0}.get(k, 1.0)
        gain[a:b] = 0.0 if k == "diffuse" else 1.0
    Q, K, V = (torch.empty((h, n, D), dtype=torch.bfloat16, device="cuda") for h in (hq, hkv, hkv))
    for g in range(hkv):
        u = _unit(gen, lo)
        v = _unit(gen, lo)
        v = v - (v @ u) * u
        v = v / v.norm()
        kr = torch.randn((n, D), generator=gen, device="cuda")
        b_s, b_v = top - math.log(4.0) + jit(0.3) + grow, top - math.log(8.0) + jit(0.3) + grow
        b_t = top - 4.4 + jit(0.3)
        sink, vert = torch.zeros(n, 1, device="cuda"), torch.zeros(n, 1, device="cuda")
        needles = {}
        for s, (a, b, k) in enumerate(zip(bounds[:-1], bounds[1:], kinds)):
            if k == "planted":
                sink[:4] = b_s * sd / resp
                vert[torch.tensor(r.sample(range(a + 4, b - 64), 8), device="cuda")] = b_v * sd / resp
            elif k == "delimiter":
                vert[a:b:257] = b_v * sd / resp
            elif k == "needle":
                nv = torch.randn((16, D), generator=gen, device="cuda")
                kr[torch.tensor(r.sample(range(a, b - 64), 128), device="cuda")] = nv.repeat(8, 1)
                needles[s] = nv
        E = torch.randn((24, D), generator=gen, device="cuda")
        E[:, :lo] = 0.0
        E = E / E.norm(dim=1, keepdim=True)
        topic = E[torch.tensor([r.randrange(24) for _ in range((n + 255) // 256)], device="cuda").repeat_interleave(256)[:n]]
        tk = math.sqrt(b_t * sd)
        k = kr + sink * u + vert * v + tk * topic
        k[:, :lo] += amp * table
        K[g] = k
        V[g] = torch.randn((n, D), generator=gen, device="cuda")
        for h in range(g * group, (g + 1) * group):
            kind, lam = heads[h]
            ds, dv, _, dt = drop[kind]
            q = torch.randn((n, D), generator=gen, device="cuda") * (1.0 if kind == "diffuse" else 0.25)
            q += gain * (resp * (b_s - ds + jit()) / b_s) * u + gain * (resp * (b_v - dv + jit()) / b_v) * v
            if dt is not None:
                q += tk * (b_t - dt + jit()) / b_t * topic
            q[:, :lo] += boosts[h] / mean_boost * amp * table
            for s, (a, b, k) in enumerate(zip(bounds[:-1], bounds[1:], kinds)):
                q[a:b] += {"local": 1.0, "diffuse": 0.0}.get(k, lam) * kr[a:b]
                if s in needles:
                    q[b - 64:b] += 0.5 * needles[s].repeat(4, 1)
            Q[h] = q
    return Q, K, V


# ------------------------------------------------------------------------------------------------------- state
def prepare(case, seed):
    gen, r = torch.Generator(device="cuda").manual_seed(seed), random.Random(seed)
    n, hq, hkv = case["n"], case["hq"], case["hkv"]
    p = rs.Problem(hq, hkv, n, _bounds(n, case["segments"]))
    state = {"kind": case["kind"], "p": p}
    if case["kind"] == "hidden":
        dm = case["d_model"]
        state["X"] = torch.randn((n, dm), generator=gen, device="cuda").to(torch.bfloat16)
        state["W"] = (torch.randn(((hq + 2 * hkv) * D, dm), generator=gen, device="cuda") / math.sqrt(dm)).to(torch.bfloat16)
        inv = 500000.0 ** (-torch.arange(0, D, 2, device="cuda", dtype=torch.float64) / D)
        ang = torch.arange(n, device="cuda", dtype=torch.float64)[:, None] * inv[None, :]
        state["cos"], state["sin"] = torch.cos(ang).float().contiguous(), torch.sin(ang).float().contiguous()
        state["layer"] = rs.RoutedPrefillLayer(p, None, rs.RouteConfig(budget_frac=0.15, cert_max=0.05))
        return state
    state["Q"], state["K"], state["V"] = (_planted if case["recipe"] == "planted" else _archetypes)(case, gen, r)
    dtype = torch.float32 if case["out"] == "fp32" else torch.bfloat16
    if case["kind"] == "dense":
        state["O"] = torch.empty((hq, n, D), dtype=dtype, device="cuda")
        state["lse"] = torch.empty((hq, n), dtype=torch.float32, device="cuda")
        state["onorm"] = torch.empty_like(state["lse"])
        state["ws"], state["status"] = rs.new_workspace(p, None), rs.new_status()
        return state
    cert = case["cert"] if case["cert"] >= 0.0 else None
    cfg = rs.RouteConfig(budget_frac=case["budget"], cert_max=cert, mixture_u=case["mixture"], mixture_lists=case["mixture"])
    layer = rs.RoutedPrefillLayer(p, LIBRARIES[case["library"]], cfg, out_dtype=dtype)
    state["layer"], state["fixed"] = layer, None
    if case["routes"] == "fixed":                 # 30 % A-shape, 30 % vertical-slash, 30 % block-sparse, the rest dense
        k = int(0.3 * hq)
        dense = max(1, hq // 10)
        pool = [0] * (hq - 2 * k - dense) + [1] * k + [2] * k + [3] * dense
        state["fixed"] = torch.tensor(r.sample(pool, hq), dtype=torch.int32, device="cuda")
    if case["kind"] == "graph":
        own = [state[x].clone() for x in "QKV"]   # the buffers the graph reads; every pass copies its inputs there
        state["graph"] = rs.GraphedPrefill(layer, *own)
    return state


def run(state):
    kind = state["kind"]
    if kind == "dense":
        rs.rs_dense_prefill_attn(state["p"], state["Q"], state["K"], state["V"], state["O"], state["lse"], state["onorm"], None,
                                 state["ws"], state["status"])
        return {k: state[k] for k in ("O", "lse", "onorm")}
    layer = state["layer"]
    if kind == "hidden":
        O = layer.forward_from_hidden(state["X"], state["W"], state["cos"], state["sin"])
    elif kind == "graph":
        O = state["graph"].run(state["Q"], state["K"], state["V"])
    else:
        O = layer.forward(state["Q"], state["K"], state["V"], fixed_choice=state["fixed"])
    # the retained mass m stands for the certificate: 2 (1 - m) V_max is all cancellation where a head is dense
    return {"O": O, "lse": layer.lse_sel, "onorm": layer.onorm, "choice": layer.choice, "lse_probe": layer.lse_probe,
            "vmax": layer.vmax, "m_row": layer.m_row, "m_head": layer.m_head}


# ------------------------------------------------------------------------------------------------------- work, tolerance
def _pairs(pattern, b0, b1, n):
    """Query-key pairs of one head of n rows under a pattern (block-sparse and vertical-slash: at most the budget per row)."""
    dense = n * (n + 1) // 2
    if pattern == rs.RS_DENSE:
        return dense
    per_row = {rs.RS_A_SHAPE: b0 + b1, rs.RS_VERTICAL_SLASH: b0 + b1, rs.RS_BLOCK_SPARSE: 64 * b0}[pattern]
    return dense if per_row >= n else per_row * n - per_row * per_row // 2


def work(case):
    n, hq, hkv = case["n"], case["hq"], case["hkv"]
    out = 4 if case.get("out") == "fp32" else 2
    dense = 512 * hq * (n * (n + 1) // 2)
    moved = n * D * (2 * hq + 4 * hkv) + n * hq * (out * D + 8)        # Q, K, V in; O and two fp32 words per row out
    if case["kind"] == "dense":
        return {"bytes": moved, "flops": dense}
    probe = 256 * 64 * hq * sum(_bounds(n, case["segments"])[1:])       # the probe rows against every key they may see
    if case["kind"] == "hidden":                                        # no structure in these inputs: every head ends with all keys
        dm, width = case["d_model"], (hq + 2 * hkv) * D
        return {"bytes": 2 * dm * (n + width) + n * (hq * (2 * D + 8) + 512), "flops": 2 * n * dm * width + probe + dense}
    if case["routes"] == "fixed":
        k = int(0.3 * hq)
        d = max(1, hq // 10)
        counts = [hq - 2 * k - d, k, k, d]
        attn = 512 * sum(c * _pairs(*cand, n) for c, cand in zip(counts, LIBRARIES["fixed"]))
    else:
        attn = case["budget"] * dense                                   # what the layer budget leaves to the attention
    return {"bytes": moved, "flops": probe + attn}


def tolerance(case):
    # Against 64-bit attention of the same inputs (bf16 probabilities, fp32 accumulation) a 4K dense pass differs by 1.9e-3
    # with bf16 output and 1.0e-3 with fp32 output in the 2-norm, and nowhere by more than 1e-2 of the value or the root mean
    # square; four times that.  Routes are whole numbers and stay what they are.
    return {"rel": 4e-3 if case.get("out") == "fp32" else 8e-3, "max": 0.04}


# ------------------------------------------------------------------------------------------------------- 64-bit results
def _attend(q, k, v, keep=None, step=1024):
    """Causal attention of one head in 64 bits: O [n, d] and the log-sum-exp of every row; keep(rows, keys) narrows the mask."""
    n = q.shape[0]
    O, lse = torch.empty_like(q), torch.empty(n, dtype=q.dtype, device=q.device)
    for a in range(0, n, step):
        b = min(n, a + step)
        rows, keys = torch.arange(a, b, device=q.device)[:, None], torch.arange(b, device=q.device)[None, :]
        mask = rows >= keys
        if keep is not None:
            mask &= keep(rows, keys)
        x = (q[a:b] @ k[:b].T / math.sqrt(D)).masked_fill_(~mask, -math.inf)
        lse[a:b] = torch.logsumexp(x, dim=1)
        O[a:b] = torch.exp_(x.sub_(lse[a:b, None])) @ v[:b]
    return O, lse


def _probe_rows(q, k, q1):
    """Probability rows and log-sum-exps of the 64 queries in front of q1."""
    rows, keys = torch.arange(q1 - 64, q1, device=q.device)[:, None], torch.arange(q1, device=q.device)[None, :]
    x = (q[q1 - 64:q1] @ k[:q1].T / math.sqrt(D)).masked_fill_(rows < keys, -math.inf)
    lse = torch.logsumexp(x, dim=1)
    return torch.exp(x - lse[:, None]), lse


def _vertical_slash(P, n, n_cols, n_offs):
    """keep() of the vertical-slash pattern ranked by the probe rows P: the heaviest columns, and the block diagonals that the
    offset 0 and the heaviest other offsets touch."""
    offs = (torch.arange(n - 64, n, device=P.device)[:, None] - torch.arange(n, device=P.device)[None, :])
    slash = torch.zeros(n, dtype=P.dtype, device=P.device).index_add_(0, offs.clamp_(min=0).flatten(), P.flatten())
    slash[0] = math.inf
    top = lambda x, count: torch.sort(x, descending=True, stable=True).indices[:count]
    col = torch.zeros(n, dtype=torch.bool, device=P.device)
    col[top(P.sum(0), n_cols)] = True
    best = top(slash, n_offs)
    diag = torch.zeros(n // 64 + 2, dtype=torch.bool, device=P.device)
    diag[best // 64] = True
    diag[(best + 63) // 64] = True
    return lambda rows, keys: col[keys] | diag[(rows // 64 - keys // 64).clamp(min=0)]


def _project(state, hq, hkv):
    """Q, K, V of the hidden states in 64 bits: the projection, and rotate-half of Q and K."""
    n = state["X"].shape[0]
    y = (state["X"].double() @ state["W"].double().T).view(n, hq + 2 * hkv, D).transpose(0, 1)
    cos, sin = (torch.cat([state[x].double()] * 2, dim=1) for x in ("cos", "sin"))
    rotated = torch.cat([-y[..., D // 2:], y[..., :D // 2]], dim=-1)
    qk = y * cos + rotated * sin
    return qk[:hq], qk[hq:hq + hkv], y[hq + hkv:]


def _all_or_little(n):
    """No window or block budget of the online library covers nearly all keys of n without covering all of them."""
    return not any(w < n <= 1.25 * w for w in (1024, 2048, 4096, 8192, 3200, 6400, 12800, 25600))


def exact(case, seed):
    """What run() returns in 64 bits.  Attention outputs where the executed mask is known without the router: dense, the layer
    from hidden states (without structure every head ends with all keys), and the one-head library, whose budget takes its
    vertical-slash candidate.  Elsewhere what the probe gives: its log-sum-exps and the largest value norms."""
    state = prepare(case, seed)
    kind, hq, hkv = case["kind"], case["hq"], case["hkv"]
    group, bounds = hq // hkv, _bounds(case["n"], case["segments"])
    Q, K, V = _project(state, hq, hkv) if kind == "hidden" else (state[x] for x in "QKV")
    one_head = case.get("library") == "one_head"
    full = kind == "dense" or one_head or kind == "hidden" and _all_or_little(case["n"])
    O, lse, probe = [], [], []
    for h in range(hq):
        q, k, v = Q[h].double(), K[h // group].double(), V[h // group].double()
        rows = [_probe_rows(q, k, q1) for q1 in bounds[1:]] if kind != "dense" else []
        probe.append([r[1] for r in rows])
        if full:
            keep = _vertical_slash(rows[0][0], case["n"], 256, 512) if one_head else None
            o, l = _attend(q, k, v, keep)
            O.append(o.float())
            lse.append(l)
    out = {"O": None, "lse": None, "onorm": None}
    if full:
        O, lse = torch.stack(O), torch.stack(lse)
        out = {"O": O, "lse": lse, "onorm": torch.linalg.vector_norm(O, dim=-1, dtype=torch.float64)}
    if kind == "dense":
        return out
    norms = torch.stack([torch.linalg.vector_norm(v.double(), dim=-1) for v in V])
    lse_probe = torch.stack([torch.stack(x) for x in probe])
    out.update(choice=None, lse_probe=lse_probe, vmax=torch.stack([norms[:, :q1].amax(1) for q1 in bounds[1:]]), m_row=None, m_head=None)
    if full:
        m = torch.exp(lse[:, -64:] - lse_probe[:, 0]).clamp(max=1.0)
        out.update(m_row=m, m_head=m.mean(1))
    return out
