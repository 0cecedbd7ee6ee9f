"""What a program that serves a LiSA model has this library do, as cases that can be timed and compared.

Each case is a dict of plain values; `prepare` makes what such a program has in hand before the call (inputs from a seed,
weights, caches, workspaces), `run` makes ONE pass through the binding's entry points.  The shapes are those of the
workloads in paper_2408_01890_b200/synth.py, of the paper's own default layer (concatenating Integrate, 64 x 256 and
256 x 32, r = 20), and generic prompt and context lengths.  Four kinds:

  decode   one new token per sequence through an anchor layer (optional) and the `chain` shared layers behind it: per layer
           the cache append and the attention call (and, with "project", the projections either side of it); score rows are
           handed from layer to layer.  "graph": the step is captured in a CUDA graph once and replayed, as a serving loop does.
  prefill  a prompt through the same layers.  via "carry": anchor attention, then layer by layer with carried scores;
           via "recompute": anchor attention, then every shared layer from the anchor's q0, k0; via "layer": the deepest
           shared layer alone.  With "append" every layer's cache is filled as well.
  project  a prompt's hidden states through a shared layer's [W_Q' | W_K' | W_V] and through W_O.
"""
from __future__ import annotations

import math

import torch

from paper_2408_01890_b200 import binding as lb

D = 128  # head width of every LLaMA shape here
L7 = {"Hq": 32, "Hkv": 32, "r": 21, "m": 64, "act": "relu", "integrate": "add"}     # LLaMA2-7B-shaped
L8 = {"Hq": 32, "Hkv": 8, "r": 21, "m": 64, "act": "relu", "integrate": "add"}      # LLaMA3-8B-shaped (grouped queries)
L13 = {"Hq": 40, "Hkv": 40, "r": 21, "m": 80, "act": "relu", "integrate": "add"}    # LLaMA2-13B-shaped
LP = {"Hq": 32, "Hkv": 32, "r": 20, "m": 256, "act": "relu", "integrate": "concat"}  # the paper's default layer


def _decode(model, B, L, chain, anchor=True, ragged=False, rows="f32", project=False, graph=False, **name):
    return dict(name, kind="decode", **model, d=D, B=B, L=L, chain=chain, anchor=anchor, ragged=ragged, rows=rows,
                project=project, graph=graph, dtype="bf16")


def _prefill(model, B, N, chain, via="carry", anchor=True, append=True, dtype="bf16", d=D, **name):
    return dict(name, kind="prefill", **model, d=d, B=B, N=N, chain=chain, via=via, anchor=anchor, append=append, dtype=dtype)


def _project(model, B, N, **name):
    return dict(name, kind="project", **model, d=D, B=B, N=N, dtype="bf16")


def listed():
    return [
        # one user's chat turn: a single sequence, a short context, call by call from Python, projections included
        _decode(L7, 1, 333, 3, project=True, name="decode_one_sequence"),
        # continuous batching: sequences of every length in one call, grouped queries, 2-byte score rows
        _decode(L8, 16, 2900, 3, ragged=True, rows="bf16", name="decode_8b_ragged"),
        # a large uniform batch, one shared layer of the 13B shape: the HBM-bound case
        _decode(L13, 64, 4096, 1, anchor=False, name="decode_13b_layer"),
        # a step of the 7B-shaped stack (anchor + three shared layers, projections included) replayed from a graph
        _decode(L7, 32, 2176, 3, project=True, graph=True, name="decode_7b_step"),
        # the paper's default model (concatenating aligner, hidden width 256), a modest batch
        _decode(LP, 8, 1111, 2, name="decode_paper_default"),
        # the parity workload in fp32: a tiny layer, where launches and latency count
        _prefill({"Hq": 4, "Hkv": 4, "r": 8, "m": 16, "act": "relu", "integrate": "add"}, 1, 128, 1, via="recompute",
                 append=False, dtype="f32", d=32, name="prefill_tiny_f32"),
        # a chat prompt of an odd length through an anchor and its chain
        _prefill(L8, 1, 197, 3, name="prefill_short"),
        # a 7B-shaped shared layer over one prompt (SiLU), recomputed from its anchor
        _prefill(dict(L7, act="silu"), 1, 2048, 1, via="layer", anchor=False, append=False, name="prefill_7b_layer"),
        # the paper's default layer over one prompt
        _prefill(LP, 1, 2048, 1, name="prefill_paper_default"),
        # 40 heads, two prompts of an odd length
        _prefill(L13, 2, 1777, 2, name="prefill_13b_ragged"),
        # long documents: the 8B-shaped anchor and its chain of three, the largest case
        _prefill(L8, 4, 8192, 3, name="prefill_8b_chain"),
        # the projections of a 7B-shaped shared layer over a batch of prompts
        _project(L7, 8, 2048, name="project_prompts"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    what = rng.choice(["decode", "decode", "decode", "decode", "decode", "prefill", "prefill", "prefill", "prefill", "prefill", "tiny", "project"])
    if what == "decode":
        model = dict(rng.choice([L7, L8, L13, LP]))
        if model["integrate"] == "add":
            model["act"] = rng.choice(["relu", "relu", "silu"])
        B, chain, anchor = _log(rng, 1, 64), rng.randint(1, 3), rng.random() < 0.75
        layers = chain + (1 if anchor else 0)
        most = 262144 // (layers if model["Hkv"] > 8 else 1)       # cached positions: the 13B-shaped case's, over all layers
        if model["integrate"] == "concat":
            most //= 4
        return _decode(model, B, _log(rng, 16, max(32, min(8192, most // B))), chain, anchor, ragged=rng.random() < 0.4,
                       rows=rng.choice(["f32", "f32", "bf16"]), project=rng.random() < 0.4, graph=rng.random() < 0.4)
    if what == "prefill":
        model = dict(rng.choice([L7, L8, L13, LP]))
        if model["integrate"] == "add":
            model["act"] = rng.choice(["relu", "relu", "silu"])
        B, chain = rng.randint(1, 4), rng.randint(1, 3)
        via = rng.choice(["carry", "carry", "layer"])
        # positions x heads x links, against the largest listed case
        cost = B * model["Hq"] * (chain + 1) * (3 if model["integrate"] == "concat" else 1) * (2 if via == "layer" else 1)
        most = int(math.sqrt(4 * 32 * 4 * 8192.0 ** 2 / cost))
        return _prefill(model, B, _log(rng, 33, min(8192, most)), chain, via, anchor=via == "carry", append=via == "carry")
    if what == "tiny":
        heads = rng.choice([2, 4, 8])
        model = {"Hq": heads, "Hkv": rng.choice([1, heads]), "r": rng.randint(4, 12), "m": 4 * heads, "act": "relu", "integrate": "add"}
        return _prefill(model, rng.randint(1, 2), _log(rng, 16, 200), rng.randint(1, 2), via="recompute", append=False, dtype="f32",
                        d=rng.choice([32, 64]))
    return _project(rng.choice([L7, L8, L13]), rng.randint(1, 8), _log(rng, 4, 2048))


# ------------------------------------------------------------------------------------------------------------------
def _dtype(c):
    return torch.bfloat16 if c["dtype"] == "bf16" else torch.float32


class _Rng:
    """N(0, std^2) tensors on the GPU, one after the other from a seed."""

    def __init__(self, seed):
        self.g = torch.Generator(device="cuda")
        self.g.manual_seed(int(seed) * 2654435761 % (1 << 62))

    def normal(self, shape, dtype, std=1.0):
        x = torch.randn(tuple(shape), generator=self.g, device="cuda", dtype=dtype)
        return x if std == 1.0 else x.mul_(std)


def _aligner(c, rng):
    h_in = c["Hq"] * (2 if c["integrate"] == "concat" else 1)
    return (rng.normal((h_in, c["m"]), _dtype(c), h_in ** -0.5), rng.normal((c["m"], c["Hq"]), _dtype(c), c["m"] ** -0.5))


def _link(c, qp, kp, w):
    return lb.Link(qp, kp, w[0], w[1], act=lb.ACTS[c["act"]],
                   integrate=lb.INTEGRATE_CONCAT if c["integrate"] == "concat" else lb.INTEGRATE_ADD)


def _lengths(c, seed):
    """Context lengths of a decode batch, the new token included: all L, or spread over [L/8, L]."""
    if not c["ragged"]:
        return [c["L"]] * c["B"]
    g = torch.Generator().manual_seed(int(seed))
    lens = torch.randint(max(1, c["L"] // 8), c["L"] + 1, (c["B"],), generator=g).tolist()
    lens[0] = c["L"]
    return lens


def _prepare_decode(c, seed):
    rng, dt = _Rng(seed), _dtype(c)
    B, L, Hq, Hkv, d, r = c["B"], c["L"], c["Hq"], c["Hkv"], c["d"], c["r"]
    L_cap, dm = (L + 64 + 7) // 8 * 8, Hq * d
    s = {"c": c, "layers": []}
    for l in range(c["chain"] + (1 if c["anchor"] else 0)):
        std = c["anchor"] and l == 0
        cache = lb.KVCacheLayer(lb.CACHE_STANDARD if std else lb.CACHE_SHARED, B, Hkv, L_cap, d, 0 if std else r, dtype=dt)
        cache.k.normal_(generator=rng.g)
        cache.v.normal_(generator=rng.g)
        y = {"std": std, "cache": cache, "k_new": rng.normal((B, 1, Hkv, d if std else r), dt), "v_new": rng.normal((B, 1, Hkv, d), dt),
             "a": rng.normal((B, 1, Hq, d if std else r), dt), "out": torch.zeros((B, 1, Hq, d), dtype=dt, device="cuda")}
        if not std:
            y["w"] = _aligner(c, rng)
        if c["project"]:
            n = Hq * (d if std else r) + Hkv * (d if std else r) + Hkv * d
            y["h"] = rng.normal((B, 1, dm), dt)
            y["w_in"], y["w_o"] = rng.normal((dm, n), dt, dm ** -0.5), rng.normal((dm, dm), dt, dm ** -0.5)
            y["y"] = torch.zeros((B, 1, 1, dm), dtype=dt, device="cuda")
        s["layers"].append(y)
    lens = torch.tensor(_lengths(c, seed), dtype=torch.int32)
    s["before"] = (lens - 1).cuda()
    s["lens"] = lens.cuda() if c["ragged"] or c["graph"] else None
    row_dt = torch.bfloat16 if c["rows"] == "bf16" else torch.float32
    # one row buffer per hand-off (row l: what layer l wrote, or the given row in front of the first layer)
    s["rows"] = [torch.zeros((B, Hq, L_cap), dtype=row_dt, device="cuda") for _ in range(len(s["layers"]) - (1 if c["anchor"] else 0))]
    if not c["anchor"]:
        s["rows"][0].normal_(generator=rng.g)
    s["ws"] = torch.empty(lb.decode_workspace_bytes(B, Hq, d, L), dtype=torch.uint8, device="cuda")
    if c["graph"]:
        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side):
            _decode_step(s)
        torch.cuda.current_stream().wait_stream(side)
        torch.cuda.synchronize()
        s["graph"] = torch.cuda.CUDAGraph()
        with torch.cuda.graph(s["graph"]):
            _decode_step(s)
    return s


def _decode_step(s):
    c, cur = s["c"], -1 if s["c"]["anchor"] else 0
    L, lens, ws, rows, n = c["L"], s["lens"], s["ws"], s["rows"], len(s["layers"])
    for l, y in enumerate(s["layers"]):
        if c["project"]:
            lb.lisa_project(y["h"], y["w_in"], [y["a"], y["k_new"], y["v_new"]])
        lb.lisa_kvcache_append(y["cache"], y["k_new"], y["v_new"], s["before"])
        row_out = rows[cur + 1] if l + 1 < n else None
        if y["std"]:
            lb.lisa_attn_anchor(y["a"], cache=y["cache"], L=L, seq_lens=lens, out=y["out"], out_scores=row_out, workspace=ws)
        else:
            lb.lisa_attn_shared_decode(rows[cur], _link(c, y["a"], None, y["w"]), y["cache"], L=L, seq_lens=lens, out=y["out"],
                                       out_scores=row_out, workspace=ws)
        if c["project"]:
            lb.lisa_project(y["out"].view(c["B"], 1, -1), y["w_o"], [y["y"]])
        cur += 1


def _run_decode(s):
    if s["c"]["graph"]:
        s["graph"].replay()
    else:
        _decode_step(s)
    ys = s["layers"]
    out = {"o": [y["out"] for y in ys], "k": [y["cache"].k for y in ys], "v": [y["cache"].v for y in ys], "rows": s["rows"]}
    if s["c"]["project"]:
        out["y"] = [y["y"] for y in ys]
    return out


def _prepare_prefill(c, seed):
    rng, dt = _Rng(seed), _dtype(c)
    B, N, Hq, Hkv, d, r = c["B"], c["N"], c["Hq"], c["Hkv"], c["d"], c["r"]
    new = lambda: torch.zeros((B, N, Hq, d), dtype=dt, device="cuda")  # noqa: E731
    s = {"c": c, "q0": rng.normal((B, N, Hq, d), dt), "k0": rng.normal((B, N, Hkv, d), dt), "layers": [], "caches": []}
    if c["anchor"]:
        s["v0"], s["o0"] = rng.normal((B, N, Hkv, d), dt), new()
    for _ in range(c["chain"]):
        s["layers"].append({"qp": rng.normal((B, N, Hq, r), dt), "kp": rng.normal((B, N, Hkv, r), dt), "v": rng.normal((B, N, Hkv, d), dt),
                            "w": _aligner(c, rng), "out": new()})
    if c["append"]:
        L_cap = (N + 64 + 7) // 8 * 8
        s["caches"] = [lb.KVCacheLayer(lb.CACHE_SHARED, B, Hkv, L_cap, d, r, dtype=dt) for _ in s["layers"]]
        if c["anchor"]:
            s["caches"].insert(0, lb.KVCacheLayer(lb.CACHE_STANDARD, B, Hkv, L_cap, d, dtype=dt))
    ys = s["layers"]
    links = [_link(c, y["qp"], y["kp"], y["w"]) for y in ys]
    if c["via"] == "carry":
        s["scores"] = torch.empty(lb.lisa_prefill_scores_bytes(B, N, Hq), dtype=torch.uint8, device="cuda")
        s["ws"] = lb.prefill_carry_workspace(s["q0"], s["k0"], links[0], ys[0]["v"], ys[0]["out"], s["scores"])
    else:
        s["ws"] = lb.prefill_workspace(s["q0"], s["k0"], links, ys[-1]["v"], ys[-1]["out"])
    return s


def _run_prefill(s):
    c, ys, caches, ws = s["c"], s["layers"], s["caches"], s["ws"]
    q0, k0 = s["q0"], s["k0"]
    if c["anchor"]:
        lb.lisa_attn_anchor(q0, k0, s["v0"], out=s["o0"])
        if c["append"]:
            lb.lisa_kvcache_append(caches[0], k0, s["v0"])
    links = []
    for i, y in enumerate(ys):
        links.append(_link(c, y["qp"], y["kp"], y["w"]))
        if c["via"] == "carry":
            lb.lisa_attn_shared_prefill_carry(q0, k0, links[-1], y["v"], s["scores"], first=i == 0, keep=i + 1 < len(ys),
                                              out=y["out"], workspace=ws)
        elif c["via"] == "recompute" or i + 1 == len(ys):
            lb.lisa_attn_shared_prefill(q0, k0, links, y["v"], out=y["out"], workspace=ws)
        if c["append"]:
            lb.lisa_kvcache_append(caches[i + (1 if c["anchor"] else 0)], y["kp"], y["v"])
    outs = [y["out"] for y in ys] if c["via"] != "layer" else [ys[-1]["out"]]
    if c["anchor"]:
        outs.insert(0, s["o0"])
    return {"o": outs, "k": [x.k for x in caches], "v": [x.v for x in caches]}


def _prepare_project(c, seed):
    rng, dt = _Rng(seed), _dtype(c)
    B, N, Hq, Hkv, d, r = c["B"], c["N"], c["Hq"], c["Hkv"], c["d"], c["r"]
    dm = Hq * d
    new = lambda H, x: torch.zeros((B, N, H, x), dtype=dt, device="cuda")  # noqa: E731
    return {"c": c, "h": rng.normal((B, N, dm), dt), "o": rng.normal((B, N, dm), dt),
            "w_in": rng.normal((dm, Hq * r + Hkv * r + Hkv * d), dt, dm ** -0.5), "w_o": rng.normal((dm, dm), dt, dm ** -0.5),
            "outs": [new(Hq, r), new(Hkv, r), new(Hkv, d)], "y": new(1, dm)}


def _run_project(s):
    lb.lisa_project(s["h"], s["w_in"], s["outs"])
    lb.lisa_project(s["o"], s["w_o"], [s["y"]])
    return {"outs": s["outs"], "y": s["y"]}


def prepare(case, seed):
    return {"decode": _prepare_decode, "prefill": _prepare_prefill, "project": _prepare_project}[case["kind"]](case, seed)


def run(state):
    return {"decode": _run_decode, "prefill": _run_prefill, "project": _run_project}[state["c"]["kind"]](state)


# ------------------------------------------------------------------------------------------------------------------
def work(case):
    """Each input read once, each output written once; the matrix products, counted two per multiply-add."""
    c = case
    B, Hq, Hkv, d, r, m = c["B"], c["Hq"], c["Hkv"], c["d"], c["r"], c["m"]
    e = 2 if c["dtype"] == "bf16" else 4
    h_in = Hq * (2 if c["integrate"] == "concat" else 1)
    ffn = 2 * h_in * m + 2 * m * Hq               # aligner, per position
    dm = Hq * d
    n_shared = Hq * r + Hkv * r + Hkv * d         # columns of a shared layer's input projection
    if c["kind"] == "project":
        rows = B * c["N"]
        return {"bytes": e * (rows * (2 * dm + n_shared + dm) + dm * (n_shared + dm)), "flops": 2 * rows * dm * (n_shared + dm)}
    if c["kind"] == "decode":
        mean = (c["L"] // 8 + c["L"]) / 2 if c["ragged"] else c["L"]
        pos = B * mean
        re = 2 if c["rows"] == "bf16" else 4
        shared = c["chain"]
        layers = shared + (1 if c["anchor"] else 0)
        by = pos * (shared * (Hkv * (r + d) * e + Hq * re) + (layers - 1) * Hq * re)   # caches, rows in, rows out (not the last layer's)
        fl = pos * shared * (2 * Hq * r + ffn + 2 * Hq * d)
        if c["anchor"]:
            by += pos * 2 * Hkv * d * e
            fl += pos * 4 * Hq * d
        by += layers * B * e * (2 * Hq * d + 2 * Hkv * d) + shared * (h_in + Hq) * m * e
        if c["project"]:
            n = shared * (n_shared + dm) + (dm + 2 * Hkv * d + dm if c["anchor"] else 0)
            by += e * (dm * n + B * n)
            fl += 2 * B * dm * n
        return {"bytes": int(by), "flops": int(fl)}
    N = c["N"]
    pos = B * N * (N + 1) // 2
    rows = B * N * e
    chain = c["chain"]
    n_out = 1 if c["via"] == "layer" else chain
    by = rows * ((Hq + Hkv) * d + chain * (Hq + Hkv) * r + n_out * (Hkv + Hq) * d)
    fl = pos * (2 * Hq * d + chain * (2 * Hq * r + ffn) + n_out * 2 * Hq * d)
    if c["anchor"]:
        by += rows * (Hkv + Hq) * d
        fl += pos * 2 * Hq * d
    if c["append"]:
        by += rows * (chain * Hkv * (r + d) + (2 * Hkv * d if c["anchor"] else 0))
    return {"bytes": int(by), "flops": int(fl)}


def tolerance(case):
    """fp32: sums of up to a few thousand terms in another order.  bf16: outputs rounded to 8 mantissa bits, probabilities and
    scores rounded to 8-11 bits on the way; a projection rounds only its result."""
    if case["dtype"] == "f32":
        return {"rel": 1e-5, "max": 1e-3}
    return {"rel": 2e-3} if case["kind"] == "project" else {"rel": 1e-2}
