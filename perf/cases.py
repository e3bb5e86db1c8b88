"""Timed work of the library through its public entry points (paper_2510_19705_b200.binding).

Sizes are those of inputs.WORKLOADS, of bench.py's options (--batch 8, --search-hierarchy) and of the tests.

Generation cases run hsd_generate with the decision log on, because that is the entry point's way of giving
logits beside tokens.  Bf16 models fix the accept decisions with hsd_set_iid_acceptance (as bench.py --coin
does): the coins are keyed by position and not by logits, so every build runs the same passes over the same
number of rows, and the counters have to agree exactly.  Such a case returns those counters and, per sequence and
level, the logits of the first position the level evaluates after the prompt: these depend on the prompt alone.
Everything later is conditioned on sampled tokens, which another correct rounding of a bf16 logit may sample
differently.  The fp32 model runs the real accept rule and returns its tokens as well.
"""
import math
import os
import random
import tempfile

import numpy as np
import torch

from paper_2510_19705_b200 import binding, inputs

ACCEPT = 0.5            # coin of every level: near what the random-init models measure (0.49 - 0.6)


def listed():
    return [
        # smallest calls: a four-layer fp32 hierarchy; launches and host round trips are everything
        dict(name="generate_tiny_fp32", kind="generate", model="tiny3", batch=1, prompt=16, n_new=64, T="3,2", page=16),
        # a 1B-shape hierarchy, short prompt, one user
        dict(name="generate_1b", kind="generate", model="1b3", batch=1, prompt=512, n_new=64, T="4,2", page=16),
        # bench.py's default shape: one summarisation request (prompt of 1024) at the draft lengths its search picks
        dict(name="generate_8b", kind="generate", model="8b3", batch=1, prompt=1024, n_new=128, T="1,1", page=16),
        # bench.py --batch 8: eight requests of which each asks for a short answer
        dict(name="generate_8b_batch8", kind="generate", model="8b3", batch=8, prompt=1024, n_new=32, T="1,1", page=16),
        # the long-context hierarchy: two documents of 8192 tokens, a short summary each
        dict(name="generate_8b_long", kind="generate", model="8b4long", batch=2, prompt=8192, n_new=32, T="2,2,3", page=16),
        # hierarchy search (bench.py --search-hierarchy): logits of every exit layer at 128 positions ...
        dict(name="layer_logits_8b", kind="layers", model="8b3", n_tokens=128, first=1, step=1),
        # ... and the acceptance rates between all of them at 256 positions
        dict(name="alpha_32_exits", kind="alpha", models=32, rows=256, vocab=32000, dtype="bf16"),
        # one decision of a single request's round
        dict(name="verify_one", kind="verify", batch=1, t=3, vocab=32000, dtype="bf16"),
        # bench.py --workload accept
        dict(name="verify_batch", kind="verify", batch=64, t=8, vocab=32000, dtype="bf16"),
        # fp32 rows of an odd vocabulary (one added token): no row after the first is aligned
        dict(name="verify_fp32_odd", kind="verify", batch=7, t=5, vocab=32001, dtype="fp32"),
        # level-0 sampling for a batch of requests
        dict(name="draft_batch", kind="draft", batch=16, rows=4, vocab=32000, dtype="bf16"),
        # one gate projection of the 8B shape at the row count of a batch-8 verification
        dict(name="gemm_gate", kind="gemm", R=24, N=14336, K=4096),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["generate", "generate", "generate", "layers", "alpha", "verify", "verify", "draft", "gemm", "gemm"])
    if kind == "generate":
        model = rng.choice(["tiny3", "1b3", "1b3", "8b3", "8b3", "8b4long"])
        levels = len(inputs.WORKLOADS[model]["exits"])
        T = ",".join(str(rng.randint(1, 3)) for _ in range(levels - 1))
        page = rng.choice([16, 16, 32, 64])
        if model == "tiny3":
            return dict(kind=kind, model=model, batch=rng.randint(1, 3), prompt=_log_int(rng, 4, 48), n_new=rng.randint(8, 64), T=T, page=page)
        if model == "1b3":
            return dict(kind=kind, model=model, batch=rng.randint(1, 4), prompt=_log_int(rng, 16, 2048), n_new=_log_int(rng, 4, 48), T=T, page=page)
        if model == "8b3":
            return dict(kind=kind, model=model, batch=rng.randint(1, 6), prompt=_log_int(rng, 32, 1400), n_new=_log_int(rng, 4, 32), T=T, page=page)
        return dict(kind=kind, model=model, batch=1, prompt=rng.randint(2049, 8192), n_new=_log_int(rng, 4, 24), T=T, page=page)
    if kind == "layers":
        model = rng.choice(["1b3", "1b3", "8b3"])
        return dict(kind=kind, model=model, n_tokens=_log_int(rng, 1, 128), first=rng.randint(1, 4), step=rng.randint(1, 5))
    if kind == "alpha":
        return dict(kind=kind, models=rng.randint(2, 32), rows=_log_int(rng, 8, 256), vocab=rng.choice([2048, 32000, 32000, rng.randint(5000, 32768)]),
                    dtype=rng.choice(["bf16", "bf16", "fp32"]))
    if kind in ("verify", "draft"):
        vocab, dtype = rng.choice([2048, 32000, 32000, rng.randint(5000, 50000)]), rng.choice(["bf16", "bf16", "fp32"])
        if kind == "verify":
            return dict(kind=kind, batch=_log_int(rng, 1, 64), t=rng.randint(1, 8), vocab=vocab, dtype=dtype)
        return dict(kind=kind, batch=_log_int(rng, 1, 64), rows=rng.randint(1, 4), vocab=vocab, dtype=dtype)
    N, K = rng.choice([(1024, 4096), (4096, 4096), (14336, 4096), (4096, 14336), (32000, 4096), (5632, 2048), (2048, 5632)])
    return dict(kind=kind, R=_log_int(rng, 1, 256), N=N - rng.choice([0, 0, rng.randint(1, 127)]), K=K)


# ------------------------------------------------------------------------------------------------ inputs
def _ints(text):
    return [int(v) for v in text.split(",")]


def _selected(case):
    return list(range(case["first"], inputs.WORKLOADS[case["model"]]["model"]["n_layers"] + 1, case["step"]))


def _accept_inputs(case, seed):
    return inputs.make_accept_logits(case["batch"], case["t"], case["vocab"], seed, device="cuda", dtype=case["dtype"])


def _alpha_logits(case, seed):
    """Logits of nested exits: one row per position plus noise that falls with depth."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    L, R, V = case["models"], case["rows"], case["vocab"]
    out = torch.empty(L, R, V, device="cuda", dtype=torch.bfloat16 if case["dtype"] == "bf16" else torch.float32)
    base = torch.randn(R, V, generator=g, device="cuda") * 3.0
    for i in range(L):
        out[i] = base + torch.randn(R, V, generator=g, device="cuda") * (1.5 * (L - 1 - i) / max(1, L - 1))
    return out


def _gemm_inputs(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    A = torch.randn(case["R"], case["K"], generator=g, device="cuda").to(torch.bfloat16)
    W = (torch.randn(case["N"], case["K"], generator=g, device="cuda") * 0.02).to(torch.bfloat16)
    return A, W


def _weights(cfg, seed):
    """inputs.make_weights with the residual stream of a trained decoder: unit-scale embeddings and the two
    projections that write to the stream scaled by 1 / sqrt(2 layers) (the usual initialisation).  With all
    matrices at one scale every layer would rewrite the stream, and one flipped bf16 rounding in the first
    layer would reach the logits at the size of their own error."""
    w = inputs.make_weights(cfg, seed, device="cuda")
    w["embed"].mul_(50.0)
    for layer in w["layers"]:
        layer["wo"].mul_((2 * cfg["n_layers"]) ** -0.5)
        layer["wd"].mul_((2 * cfg["n_layers"]) ** -0.5)
    return w


def _model_inputs(case, seed):
    wl = inputs.WORKLOADS[case["model"]]
    cfg = wl["model"]
    weights = _weights(cfg, seed)
    n, batch = (case["n_tokens"], 1) if case["kind"] == "layers" else (case["prompt"], case["batch"])
    return cfg, wl["exits"], weights, inputs.make_prompts(cfg["vocab"], batch, n, seed).cuda()


def prepare(case, seed):
    kind = case["kind"]
    if kind == "gemm":
        A, W = _gemm_inputs(case, seed)
        ws = torch.empty(binding.hsd_gemm_workspace_bytes(case["R"], case["N"], case["K"]) + 256, dtype=torch.uint8, device="cuda")
        return dict(kind=kind, A=A, W=W, ws=ws)
    if kind == "alpha":
        return dict(kind=kind, logits=_alpha_logits(case, seed))
    if kind == "verify":
        p, q = _accept_inputs(case, seed)
        ws = torch.empty(binding.hsd_verify_workspace_bytes(case["batch"], case["t"]), dtype=torch.uint8, device="cuda")
        return dict(kind=kind, p=p, q=q, x=binding.hsd_draft_sample(q, seed, 0), seed=seed, ws=ws)
    if kind == "draft":
        g = torch.Generator(device="cuda")
        g.manual_seed(seed)
        dt = torch.bfloat16 if case["dtype"] == "bf16" else torch.float32
        logits = (torch.randn(case["batch"], case["rows"], case["vocab"], generator=g, device="cuda") * 3.0).to(dt)
        return dict(kind=kind, logits=logits, seed=seed)
    cfg, exits, weights, prompt = _model_inputs(case, seed)
    if kind == "layers":
        T = [1] * (len(exits) - 1)
        eng = binding.Hsd(cfg, weights, exits, T, max_batch=1, max_seq=case["n_tokens"] + 64)
        return dict(kind=kind, eng=eng, tokens=prompt[0].contiguous(), layers=_selected(case))
    T = _ints(case["T"])
    eng = binding.Hsd(cfg, weights, exits, T, max_batch=case["batch"],
                      max_seq=case["prompt"] + case["n_new"] + sum(T) + len(exits) + 8, page_size=case["page"])
    if cfg["dtype"] == "bf16":
        eng.set_iid_acceptance([ACCEPT] * len(T))
    calls = 1                                    # log records of a sequence's first round, at most
    for t in T[1:]:
        calls = t * (calls + 1)
    folder = tempfile.TemporaryDirectory()
    return dict(kind=kind, eng=eng, prompt=prompt, n_new=case["n_new"], seed=seed, records=case["batch"] * (calls + 1),
                folder=folder, path=os.path.join(folder.name, "log"), fp32=cfg["dtype"] == "fp32")


# ------------------------------------------------------------------------------------------------ one pass
COUNTERS = ("calls", "rows", "drafted", "tested", "accepted", "emitted", "forwards")


def run(state):
    kind = state["kind"]
    if kind == "gemm":
        return binding.hsd_gemm_bf16(state["A"], state["W"], workspace=state["ws"], check=False)
    if kind == "alpha":
        return binding.hsd_pairwise_alpha(state["logits"])
    if kind == "verify":
        return binding.hsd_verify_level(1, state["p"], state["q"], state["x"], state["seed"], 0, workspace=state["ws"])
    if kind == "draft":
        return binding.hsd_draft_sample(state["logits"], state["seed"], 0)
    eng = state["eng"]
    if kind == "layers":
        return eng.layer_logits(state["tokens"], state["layers"])
    eng.set_trace(state["path"], state["records"])
    tokens, stats, _ = eng.generate(state["prompt"], state["n_new"], state["seed"])
    eng.set_trace(None)
    first = [[None] * eng.n_levels for _ in range(tokens.shape[0])]
    for rec in binding.read_trace(state["path"]):
        if rec["logits"] is not None and first[rec["seq"]][rec["level"]] is None:
            first[rec["seq"]][rec["level"]] = rec["logits"][0]
    out = {"logits": [np.stack(rows) for rows in first],
           "counters": np.array([[s[k] for k in COUNTERS] for s in stats], dtype=np.int64)}
    if state["fp32"]:
        out["tokens"] = tokens
    return out


# ------------------------------------------------------------------------------------------------ least work
def _layer_params(cfg):
    d, hd = cfg["d_model"], cfg["head_dim"]
    return d * hd * (2 * cfg["n_q_heads"] + 2 * cfg["n_kv_heads"]) + 3 * d * cfg["d_ff"]


def _passes(case, K, T):
    """Expected (forwards, rows) of every level: Algorithm 1 with coins, level-synchronous over the batch."""
    rng = random.Random(1)
    forwards, rows = [0] * (K + 1), [0] * (K + 1)
    length = [0] * case["batch"]

    def level(i, act):
        if i == 0:
            for _ in range(T[0] if T else 1):
                forwards[0] += 1
                rows[0] += len(act)
                for b in act:
                    length[b] += 1
            return
        got = {b: 0 for b in act}
        while True:
            need = [b for b in act if got[b] < (T[i] if i < K else 1)]
            if not need:
                return
            start = {b: length[b] for b in need}
            level(i - 1, need)
            forwards[i] += 1
            for b in need:
                t = length[b] - start[b]
                rows[i] += t + 1
                n = 0
                while n < t and rng.random() < ACCEPT:
                    n += 1
                length[b] = start[b] + n + 1
                got[b] += n + 1

    while True:
        act = [b for b in range(case["batch"]) if length[b] < case["n_new"]]
        if not act:
            return forwards, rows
        level(K, act)


def work(case):
    kind = case["kind"]
    es = 4 if case.get("dtype") == "fp32" else 2
    if kind == "gemm":
        R, N, K = case["R"], case["N"], case["K"]
        return {"bytes": 2 * K * (R + N) + 4 * R * N, "flops": 2 * R * N * K}
    if kind == "alpha":
        L, RV = case["models"], case["rows"] * case["vocab"]
        return {"bytes": L * RV * es, "flops": L * (L - 1) * RV}
    if kind == "verify":
        rows = case["batch"] * (2 * case["t"] + 1)
        return {"bytes": rows * case["vocab"] * es, "flops": rows * case["vocab"] * 2}
    if kind == "draft":
        n = case["batch"] * case["rows"] * case["vocab"]
        return {"bytes": n * es, "flops": n * 2}
    wl = inputs.WORKLOADS[case["model"]]
    cfg, exits = wl["model"], wl["exits"]
    es = 4 if cfg["dtype"] == "fp32" else 2
    P, head = _layer_params(cfg), cfg["vocab"] * cfg["d_model"]
    attn = 4 * cfg["n_q_heads"] * cfg["head_dim"]              # flops of one (query, key) pair of a layer
    kv = 2 * cfg["n_kv_heads"] * cfg["head_dim"] * es          # cached bytes of one position of a layer
    if kind == "layers":
        n, sel = case["n_tokens"], _selected(case)
        return {"bytes": es * (sel[-1] * P + head + len(sel) * n * cfg["vocab"]),
                "flops": 2 * n * (sel[-1] * P + len(sel) * head) + sel[-1] * attn * n * n / 2}
    B, n, K = case["batch"], case["prompt"], len(exits) - 1
    forwards, rows = _passes(case, K, _ints(case["T"]))
    nl = cfg["n_layers"]
    total = es * nl * P + B * n * nl * kv                      # the prompt: weights read once, cache written
    flops = 2 * B * n * nl * P + B * nl * attn * n * n / 2
    ctx = n + case["n_new"] / 2
    for i in range(K + 1):
        total += forwards[i] * es * (exits[i] * P + head) + forwards[i] * B * ctx * exits[i] * kv
        flops += 2 * rows[i] * (exits[i] * P + head) + rows[i] * ctx * exits[i] * attn
    return {"bytes": total, "flops": flops}


def tolerance(case):
    kind = case["kind"]
    if kind in ("verify", "draft"):
        return "exact"                                         # integer decisions on given logits
    if kind == "gemm":
        return {"rel": 1e-5, "max": 1e-4}                      # fp32 sums in another order
    if kind == "alpha":
        return {"rel": 1e-5, "max": 1e-4}                      # fp32 softmax
    if inputs.WORKLOADS[case["model"]]["model"]["dtype"] == "fp32":
        return {"rel": 1e-5, "max": 1e-4}
    # bf16 rounding points through the layers: the same rows through the generation's one-launch pass and through
    # hsd_layer_logits (other summation orders) differ by 0.0049 - 0.0058 of the norm over the exits, 0.032 at most
    return {"rel": 2e-2, "max": 1e-1}


# ------------------------------------------------------------------------------------------------ 64 bits
def _norm(x, gain, eps):
    return x * torch.rsqrt(x.square().mean(-1, keepdim=True) + eps) * gain.double()


def _attention(q, k, v, hd):
    """Causal attention; q [nq, n, hd], k / v [nkv, n, hd]; queries in blocks to bound the score matrix."""
    nq, n, _ = q.shape
    group = nq // k.shape[0]
    out = torch.empty_like(q)
    for h in range(nq):
        kt, vh = k[h // group].transpose(0, 1), v[h // group]
        for a in range(0, n, 2048):
            b = min(n, a + 2048)
            s = (q[h, a:b] @ kt[:, :b]) / math.sqrt(hd)
            mask = torch.arange(b, device=q.device)[None, :] > torch.arange(a, b, device=q.device)[:, None]
            out[h, a:b] = torch.softmax(s.masked_fill(mask, -math.inf), -1) @ vh[:b]
    return out


def _exact_forward(cfg, weights, tokens, at):
    """Logits [len(at), rows, vocab] after the layers in `at`: every position for 'layers' cases, else the last."""
    hd, nq, nkv = cfg["head_dim"], cfg["n_q_heads"], cfg["n_kv_heads"]
    layers, last_only = at
    n = tokens.shape[0]
    x = weights["embed"][tokens.long()].double()
    ang = torch.arange(n, device=x.device, dtype=torch.float64)[:, None] * \
        cfg["rope_theta"] ** (-2.0 * torch.arange(hd // 2, device=x.device, dtype=torch.float64) / hd)
    cos, sin = ang.cos()[:, None, :], ang.sin()[:, None, :]

    def rotate(t):
        a, b = t[..., :hd // 2], t[..., hd // 2:]
        return torch.cat([a * cos - b * sin, b * cos + a * sin], -1).transpose(0, 1)

    head, out = weights["lm_head"].double(), []
    for i in range(max(layers)):
        w = {k: v.double() for k, v in weights["layers"][i].items()}
        h = _norm(x, w["attn_norm"], cfg["rms_eps"])
        q, k = rotate((h @ w["wq"].T).view(n, nq, hd)), rotate((h @ w["wk"].T).view(n, nkv, hd))
        o = _attention(q, k, (h @ w["wv"].T).view(n, nkv, hd).transpose(0, 1), hd)
        x = x + o.transpose(0, 1).reshape(n, nq * hd) @ w["wo"].T
        h = _norm(x, w["mlp_norm"], cfg["rms_eps"])
        x = x + (torch.nn.functional.silu(h @ w["wg"].T) * (h @ w["wu"].T)) @ w["wd"].T
        if i + 1 in layers:
            out.append(_norm(x[-1:] if last_only else x, weights["final_norm"], cfg["rms_eps"]) @ head.T)
    return torch.stack(out)


def exact(case, seed):
    kind = case["kind"]
    if kind in ("verify", "draft"):
        return None
    if kind == "gemm":
        A, W = _gemm_inputs(case, seed)
        return A.double() @ W.double().T
    if kind == "alpha":
        logits = _alpha_logits(case, seed)
        L, R = case["models"], case["rows"]
        a = torch.zeros(L, L, dtype=torch.float64, device="cuda")
        for r in range(R):
            p = torch.softmax(logits[:, r].double(), -1)
            for i in range(L):
                a[i] += torch.minimum(p[i], p).sum(-1)
        a /= R
        a.fill_diagonal_(1.0)
        return a
    cfg, exits, weights, prompt = _model_inputs(case, seed)
    if kind == "layers":
        return _exact_forward(cfg, weights, prompt[0], (_selected(case), False))
    out = {"logits": [None] * case["batch"], "counters": None}
    for b in range(case["batch"] if case["prompt"] <= 2048 else 1):    # a long prompt: the first sequence only
        out["logits"][b] = _exact_forward(cfg, weights, prompt[b], (list(exits), True))[:, 0]
    if cfg["dtype"] == "fp32":
        out["tokens"] = None
    return out
