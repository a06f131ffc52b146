"""Measured cases of the draft-attention library: what a KV-reuse drafter calls between two target steps.

Three kinds of case, each through the package's public entry points:
  step     one drafting step (paper_2604_26412_gb300.step.DraftStep): per level of the draft chain or tree the new
           nodes' RoPE and append, then their attention over [target cache | draft K/V]; or, in "whole" mode, the
           whole chain or tree at once, as verification-shaped calls do
  fuse     the hybrid drafter's gated-delta fusion of one level's tokens
  project  the KV-only drafter's projection of one decoding step's verified tokens into the reused cache
Sizes are those of the benchmark's workloads, of the parity tests, or generic.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2604_26412_gb300 import kvshot
from paper_2604_26412_gb300 import workloads as wl
from paper_2604_26412_gb300.step import DraftStep

D = wl.HEAD_DIM
QK_EPS = 1e-6
TREE_64 = "8,12,12,12,12,8"   # 64 nodes in six levels
TREE_32 = "4,4,4,4,4,4,4,4"   # 32 nodes in eight levels


def _step(name, *, seqs=1, layers=1, min_len, max_len, levels, tree=False, page=0, hq=32, hkv=8, mode="per_depth",
          cache="bf16", qk_norm=False, lens_seed=0):
    case = {"kind": "step", "seqs": seqs, "layers": layers, "min_len": min_len, "max_len": max_len, "levels": levels,
            "tree": tree, "page": page, "hq": hq, "hkv": hkv, "mode": mode, "cache": cache, "qk_norm": qk_norm,
            "lens_seed": lens_seed}
    return {"name": name, **case} if name else case


def listed():
    return [
        # a short chat turn: every call is a few microseconds, so latency and launches are all of it
        _step("chain-1x128", min_len=128, max_len=128, levels="1,1,1,1"),
        # one conversation of ordinary length, drafted eight deep from a contiguous cache
        _step("chain-1x2k", min_len=2048, max_len=2048, levels="1,1,1,1,1,1,1,1"),
        # one long document, a tree drafter with QK-norm, a length that fills no page or tile
        _step("tree-1x20k-qknorm", min_len=20011, max_len=20011, levels=TREE_64, tree=True, page=32, qk_norm=True),
        # batched tree drafting, level by level
        _step("tree-16x4k", seqs=16, min_len=4096, max_len=4096, levels=TREE_64, tree=True, page=16),
        # the same with an fp8 target cache
        _step("tree-16x4k-fp8", seqs=16, min_len=4096, max_len=4096, levels=TREE_64, tree=True, page=16, cache="fp8"),
        # the same tree in one call (256 query rows per KV head): compute weighs as much as bandwidth
        _step("tree-16x4k-whole", seqs=16, min_len=4096, max_len=4096, levels=TREE_64, tree=True, page=16,
              mode="whole"),
        # a serving batch of mixed lengths, chain drafting
        _step("ragged-64", seqs=64, min_len=512, max_len=8192, levels="1,1,1,1,1,1,1,1", page=16, lens_seed=4),
        # the same with an fp8 target cache
        _step("ragged-64-fp8", seqs=64, min_len=512, max_len=8192, levels="1,1,1,1,1,1,1,1", page=16, cache="fp8",
              lens_seed=4),
        # long contexts, four reused target layers attended separately: the largest working set
        _step("layers-4x4x32k", seqs=4, layers=4, min_len=32768, max_len=32768, levels=TREE_32, tree=True, page=64),
        # the same with an fp8 target cache
        _step("layers-4x4x32k-fp8", seqs=4, layers=4, min_len=32768, max_len=32768, levels=TREE_32, tree=True, page=64,
              cache="fp8"),
        # fusing the two attention branches of one 12-node tree level of 16 sequences
        {"name": "fuse-192x4096", "kind": "fuse", "tokens": 192, "hidden": 4096},
        # eight verified tokens of four sequences, four sampled target layers
        {"name": "project-32x4", "kind": "project", "tokens": 32, "layers": 4, "hkv": 8, "caches": 4, "page": 64,
         "rope": True},
    ]


MAX_KEYS = 16 * 32768 * 8  # prefix keys x KV heads of the largest listed case


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step"] * 7 + ["fuse"] * 2 + ["project"])
    if kind == "fuse":
        return {"kind": "fuse", "tokens": _log_int(rng, 1, 1024), "hidden": 128 * rng.randint(8, 32)}
    if kind == "project":
        return {"kind": "project", "tokens": _log_int(rng, 1, 512), "layers": rng.randint(1, 5),
                "hkv": rng.choice([2, 4, 8, 8]), "caches": rng.randint(1, 16), "page": rng.choice([0, 16, 64]),
                "rope": rng.random() < 0.75}
    tree = rng.random() < 0.5
    if tree:
        levels, left = [], 64
        for _ in range(rng.randint(2, 8)):
            widest = min(12, left - 7, 8 * levels[-1] if levels else 12)  # a node has at most 8 children
            levels.append(rng.randint(1, widest) if left > 8 else 1)
            left -= levels[-1]
    else:
        levels = [1] * rng.randint(1, 8)
    mode = rng.choice(["per_depth", "per_depth", "per_depth", "whole"])
    hq, hkv = rng.choice([(32, 8), (32, 8), (32, 8), (32, 4), (16, 8), (64, 8)])
    seqs, layers = _log_int(rng, 1, 64), rng.choice([1, 1, 1, 2, 3, 4])
    budget = MAX_KEYS // (2 if mode == "whole" else 1)  # a whole-tree call does all levels' arithmetic at once
    max_len = _log_int(rng, 64, min(32768, max(65, budget // (seqs * layers * hkv))))
    min_len = max_len if rng.random() < 0.4 else max(1, max_len // rng.choice([2, 4, 16]))
    return _step(None, seqs=seqs, layers=layers, min_len=min_len, max_len=max_len, levels=",".join(map(str, levels)),
                 tree=tree, page=rng.choice([0, 16, 16, 32, 64, 128]), hq=hq, hkv=hkv, mode=mode,
                 cache=rng.choice(["bf16", "bf16", "fp8"]), qk_norm=rng.random() < 0.25,
                 lens_seed=rng.randrange(1 << 20))


def _spec(case) -> wl.Spec:
    n = case["seqs"] * case["layers"]
    lens = np.random.default_rng(case["lens_seed"]).integers(case["min_len"], case["max_len"], size=n, endpoint=True)
    return wl.Spec("case", case["seqs"], case["layers"], lens.tolist(), [int(x) for x in case["levels"].split(",")],
                   case["tree"], case["page"] > 0, page_size=case["page"] or 16, hq=case["hq"], hkv=case["hkv"])


def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _randn(shape, g, std=1.0):
    return (torch.randn(shape, generator=g, device="cuda") * std).to(torch.bfloat16)


def prepare(case, seed):
    if case["kind"] == "step":
        spec = _spec(case)
        inp = wl.make_inputs(spec, "cuda", seed=seed)
        fp8 = None
        if case["cache"] == "fp8":
            fp8 = (*wl.fp8_target(inp), wl.FP8_K_EXP, wl.FP8_V_EXP)
            inp.target_k, inp.target_v = fp8[0], fp8[1]  # a program with an fp8 cache keeps no bf16 one
        qk = None
        if case["qk_norm"]:
            g = _generator(seed + 1)
            w = [(0.5 + torch.rand(D, generator=g, device="cuda")).to(torch.bfloat16) for _ in range(2)]
            qk = (w[0], w[1], QK_EPS)
        return {"kind": "step", "step": DraftStep(inp, mode=case["mode"], target_fp8=fp8, qk_norm=qk)}
    g = _generator(seed)
    err = torch.zeros(1, dtype=torch.int32, device="cuda")
    if case["kind"] == "fuse":
        t, d = case["tokens"], case["hidden"]
        st = {"kind": "fuse", "n": _randn((t, d), g), "o": _randn((t, d), g),
              "w_g": _randn((d, 3 * d), g, 1.0 / math.sqrt(3 * d)), "b_g": _randn((d,), g, 0.1),
              "w_delta": _randn((d, d), g, 1.0 / math.sqrt(d)),
              "h": torch.empty((t, d), dtype=torch.bfloat16, device="cuda"), "err": err}
        desc = kvshot.make_fusion_desc(num_tokens=t, hidden=d, err_flag=err)
        size = kvshot.gated_delta_workspace_size(desc)
    else:
        t, layers, hkv, caches, page = (case[k] for k in ("tokens", "layers", "hkv", "caches", "page"))
        dkv = hkv * D
        std = 1.0 / math.sqrt(layers * dkv)
        # token t is the (t // caches)-th newly verified one of cache t % caches, at the end of its prefix
        rng = np.random.default_rng(seed)
        start = rng.integers(0, 2000, size=caches)
        idx = np.arange(t)
        cache, pos = idx % caches, start[idx % caches] + idx // caches
        cap = 2048 + -(-t // caches)
        st = {"kind": "project", "k_in": _randn((t, layers, hkv, D), g), "v_in": _randn((t, layers, hkv, D), g),
              "w_k": _randn((dkv, layers * dkv), g, std), "w_v": _randn((dkv, layers * dkv), g, std),
              "cache": torch.from_numpy(cache.astype(np.int32)).cuda(),
              "pos": torch.from_numpy(pos.astype(np.int32)).cuda(), "err": err}
        if page:
            pages = -(-cap // page)
            st["table"] = torch.from_numpy(rng.permutation(caches * pages).astype(np.int32).reshape(caches, pages)).cuda()
            shape = (caches * pages, hkv, page, D)
        else:
            st["table"] = None
            shape = (caches, hkv, cap, D)
        st["k_out"], st["v_out"] = (torch.zeros(shape, dtype=torch.bfloat16, device="cuda") for _ in range(2))
        desc = kvshot.make_project_desc(num_tokens=t, num_layers=layers, hkv=hkv, num_caches=caches, page_size=page,
                                        max_pages_per_seq=-(-cap // page) if page else 0,
                                        num_pages=shape[0] if page else 0, l_cap=0 if page else cap,
                                        rope_base=wl.ROPE_BASE, rope=case["rope"], err_flag=err)
        size = kvshot.kv_project_workspace_size(desc)
    st["workspace"] = torch.empty(size, dtype=torch.uint8, device="cuda")
    desc.workspace, desc.workspace_bytes = st["workspace"].data_ptr(), size
    st["desc"] = desc
    return st


def run(state):
    if state["kind"] == "step":
        s = state["step"]
        s.run()
        return {"out": s.out, "lse": s.lse, "q": s.q_rot, "draft_k": s.draft_k, "draft_v": s.draft_v, "err": s.err}
    if state["kind"] == "fuse":
        kvshot.gated_delta(state["desc"], state["n"], state["o"], state["w_g"], state["b_g"], state["w_delta"],
                           state["h"])
        return {"h": state["h"], "err": state["err"]}
    kvshot.kv_project(state["desc"], state["k_in"], state["v_in"], state["w_k"], state["w_v"], state["cache"],
                      state["pos"], state["table"], state["k_out"], state["v_out"])
    return {"k_out": state["k_out"], "v_out": state["v_out"], "err": state["err"]}


def work(case):
    if case["kind"] == "fuse":
        t, d = case["tokens"], case["hidden"]
        # W_g and W_delta with n, o and delta as given: 4 d^2 weights, each used once per token
        return {"bytes": 2 * (4 * d * d + d + 3 * t * d), "flops": 8 * t * d * d}
    if case["kind"] == "project":
        t, layers, dkv = case["tokens"], case["layers"], case["hkv"] * D
        return {"bytes": 2 * (2 * layers * dkv * dkv + 2 * t * layers * dkv + 2 * t * dkv) + 8 * t,
                "flops": 4 * t * layers * dkv * dkv}
    s = _spec(case)
    elem = 1 if case["cache"] == "fp8" else 2
    levels = s.levels if case["mode"] == "per_depth" else [s.n_nodes]
    total, flops, n = 0, 0, 0
    for q in levels:
        n += q
        c = s.num_caches
        total += sum(2 * s.hkv * (length * elem + n * 2) * D for length in s.seq_lens)  # K and V of the attention
        total += c * q * s.hq * (2 * D * 2 + 4)                                         # q, out, lse
        total += c * q * (2 * s.hq + 4 * s.hkv) * D * 2 + 4 * c * q                     # the append
        total += sum(4 * -(-length // s.page_size) for length in s.seq_lens) if s.paged else 0
        total += 4 * c + (4 * s.num_seqs * n if s.tree else 0)
        flops += sum(4 * s.hq * q * (length + n) * D for length in s.seq_lens)
    return {"bytes": total, "flops": flops}


def tolerance(case):
    # bf16 results of bf16 inputs with fp32 sums: each rounding of P and of the result is 2^-9 of its value
    return {"rel": 1e-2, "max": 0.1}


# ------------------------------------------------------------------ the same in 64 bits

def _rope(x, pos, base):
    """Rotate-half RoPE of x [..., 128] at positions pos (broadcast over the leading dims)."""
    freq = float(base) ** (-2.0 * torch.arange(D // 2, dtype=torch.float64, device=x.device) / D)
    ang = pos.to(torch.float64)[..., None] * freq
    c, s = ang.cos(), ang.sin()
    a, b = x[..., :D // 2], x[..., D // 2:]
    return torch.cat([a * c - b * s, b * c + a * s], dim=-1)


def _rms(x, w, eps):
    return x / torch.sqrt((x * x).mean(-1, keepdim=True) + eps) * w.to(torch.float64)


def _exact_step(case, seed):
    st = prepare(case, seed)["step"]
    inp, s = st.inp, st.inp.spec
    levels = st.levels
    c_, n_, g_ = s.num_caches, s.n_nodes, s.hq // s.hkv
    q = torch.cat(st.q_in, 1).to(torch.float64)
    k = torch.cat(st.k_in, 1).to(torch.float64)
    pos = torch.cat(st.pos, 1)
    if st.qk_norm is not None:
        wq, wk, eps = st.qk_norm
        q, k = _rms(q, wq, eps), _rms(k, wk, eps)
    q, k = _rope(q, pos[..., None], s.rope_base), _rope(k, pos[..., None], s.rope_base)
    draft_k = torch.zeros(st.draft_k.shape, dtype=torch.float64, device=q.device)
    draft_v = torch.zeros_like(draft_k)
    draft_k[:, :, :n_] = k.transpose(1, 2)
    draft_v[:, :, :n_] = torch.cat(st.v_in, 1).to(torch.float64).transpose(1, 2)
    # the append stores bf16, which is what the attention reads
    qb = q.to(torch.bfloat16).to(torch.float64)
    kb = draft_k[:, :, :n_].to(torch.bfloat16).to(torch.float64)
    parent = inp.tree_parent.cpu().numpy()
    see = np.zeros((s.num_seqs, n_, n_), bool)
    for b in range(s.num_seqs):
        for i in range(n_):
            m = i
            while m >= 0:
                see[b, i, m] = True
                m = parent[b, i] if m == i else parent[b, m]
    see = torch.from_numpy(see).to(q.device)
    out = torch.empty((c_, n_, s.hq, D), dtype=torch.float64, device=q.device)
    lse = torch.empty((c_, n_, s.hq), dtype=torch.float64, device=q.device)
    scale = 1.0 / math.sqrt(D)
    tk, tv, ks, vs = st.target_k, st.target_v, 1.0, 1.0
    if case["cache"] == "fp8":
        tk, tv = tk.view(torch.float8_e4m3fn), tv.view(torch.float8_e4m3fn)
        ks, vs = 2.0 ** wl.FP8_K_EXP, 2.0 ** wl.FP8_V_EXP
    for c in range(c_):
        length = int(s.seq_lens[c])
        mask = see[c // s.layers].repeat_interleave(g_, 0)  # rows (node, head of the group)
        for h in range(s.hkv):
            if s.paged:
                ids = inp.page_table[c, :-(-length // s.page_size)].long()
                pk = tk[:, h].view(torch.uint8 if case["cache"] == "fp8" else torch.int16)[ids]
                pv = tv[:, h].view(torch.uint8 if case["cache"] == "fp8" else torch.int16)[ids]
                pk, pv = pk.view(tk.dtype).reshape(-1, D)[:length], pv.view(tv.dtype).reshape(-1, D)[:length]
            else:
                pk, pv = tk[c, h, :length], tv[c, h, :length]
            pk, pv = pk.to(torch.float32).to(torch.float64) * ks, pv.to(torch.float32).to(torch.float64) * vs
            rows = qb[c, :, h * g_:(h + 1) * g_].reshape(n_ * g_, D) * scale
            sd = (rows @ kb[c, h].T).masked_fill(~mask, -math.inf)
            sc = torch.cat([rows @ pk.T, sd], dim=1)
            z = torch.logsumexp(sc, dim=1)
            p = torch.exp(sc - z[:, None])
            o = p[:, :length] @ pv + p[:, length:] @ draft_v[c, h, :n_]
            out[c, :, h * g_:(h + 1) * g_] = o.reshape(n_, g_, D)
            lse[c, :, h * g_:(h + 1) * g_] = z.reshape(n_, g_)
    split = lambda x: list(torch.split(x, levels, dim=1))  # noqa: E731
    return {"out": split(out), "lse": split(lse), "q": split(q), "draft_k": draft_k, "draft_v": draft_v, "err": None}


def exact(case, seed):
    if case["kind"] == "step":
        return _exact_step(case, seed)
    st = prepare(case, seed)
    f = lambda x: x.to(torch.float64)  # noqa: E731
    if case["kind"] == "fuse":
        d = case["hidden"]
        n, o = f(st["n"]), f(st["o"])
        delta, wg = o - n, f(st["w_g"])
        gate = torch.sigmoid(n @ wg[:, :d].T + o @ wg[:, d:2 * d].T + delta @ wg[:, 2 * d:].T + f(st["b_g"]))
        return {"h": n + gate * (delta @ f(st["w_delta"]).T), "err": None}
    t, hkv = case["tokens"], case["hkv"]
    k = (f(st["k_in"]).reshape(t, -1) @ f(st["w_k"]).T).reshape(t, hkv, D)
    v = (f(st["v_in"]).reshape(t, -1) @ f(st["w_v"]).T).reshape(t, hkv, D)
    pos, cache = st["pos"].long(), st["cache"].long()
    if case["rope"]:
        k = _rope(k, pos[:, None], wl.ROPE_BASE)
    k_out, v_out = f(st["k_out"]), f(st["v_out"])
    if case["page"]:
        page = st["table"][cache, pos // case["page"]].long()
        k_out[page, :, pos % case["page"]] = k
        v_out[page, :, pos % case["page"]] = v
    else:
        k_out[cache, :, pos] = k
        v_out[cache, :, pos] = v
    return {"k_out": k_out, "v_out": v_out, "err": None}
