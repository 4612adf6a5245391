"""The work that users of this library have it do, as measurable cases.

Four kinds, each through the public entry points:

  attn    tree attention of one or more layers (``adt_tree_attn``);
  draft   the growth of one draft tree: ``adt_tree_expand`` (or ``_cfg``) per
          layer, then ``adt_tree_rerank``;
  verify  the acceptance walk (``adt_tree_accept`` or ``_cfg``) and the commit
          of the accepted path's K/V (``adt_kv_compact``);
  step    a whole verify step (``verify_step.TreeVerifyStep``).

Several layers, and whole steps, are captured once in a CUDA graph and
replayed, as the decode loop and the benchmark do; single calls, the draft of
one image and the verify phase are made call by call, as the decode loop makes
them.  Lists of per-tree numbers are texts ("600,1337").
"""
from __future__ import annotations

import math

import torch

from paper_2512_21857_gb300 import binding as B
from paper_2512_21857_gb300 import synth
from paper_2512_21857_gb300.verify_step import StepShape, TreeVerifyStep

DEV = "cuda"
MODES = {"greedy": B.ACCEPT_GREEDY, "spec": B.ACCEPT_SPEC, "spec_det": B.ACCEPT_SPEC_DET}


def _ints(text):
    return [int(x) for x in str(text).split(",")]


def _text(values):
    return ",".join(str(int(v)) for v in values)


# ------------------------------------------------------------------ the cases

def listed():
    return [
        # One layer of the single verify step (8 heads x 64, KV 512, 26 nodes), called by itself:
        # what an engine that owns its layer loop calls; the smallest call.
        dict(name="attn_one_layer", kind="attn", layers=1, kv="512", nodes="26", max_nodes=26, H=8, Hkv=8, D=64,
             lmax=576, chain=False, lse=True, graph=False),
        # All layers of a LlamaGen-XL-shaped target over a 64-node tree, late in the image.
        dict(name="attn_llamagen", kind="attn", layers=36, kv="696", nodes="64", max_nodes=64, H=20, Hkv=20, D=64,
             lmax=760, chain=False, lse=False, graph=True),
        # The adjacency-adaptive ragged batch: 8 images at the 7B shape, prefixes and trees all different
        # (8 of the 32 layers).
        dict(name="attn_ragged8", kind="attn", layers=8, kv="751,1596,1444,640,1427,1245,2352,1248",
             nodes="64,64,64,27,23,7,64,64", max_nodes=64, H=32, Hkv=32, D=128, lmax=2416, chain=False, lse=False,
             graph=True),
        # Wide drafts of a LlamaGen-class model (width up to 39: more than 64 nodes), the conditional and
        # the unconditional branch of classifier-free guidance as two trees.
        dict(name="attn_wide_guided", kind="attn", layers=36, kv="693,577", nodes="192,192", max_nodes=192, H=20,
             Hkv=20, D=64, lmax=960, chain=False, lse=False, graph=True),
        # The draft head of the 7B decode loop: one layer, run once for each of a tree's growth steps, its
        # call sized for trees of up to 256 nodes while the tree holds far fewer.
        dict(name="attn_draft_head", kind="attn", layers=6, kv="1203", nodes="41", max_nodes=256, H=32, Hkv=32, D=128,
             lmax=2336, chain=False, lse=False, graph=True),
        # Grouped query heads (four to a kv head) over long prefixes, four images.
        dict(name="attn_grouped_long", kind="attn", layers=8, kv="6001,4777,3500,5120", nodes="48,64,33,60",
             max_nodes=64, H=32, Hkv=8, D=128, lmax=6144, chain=False, lse=False, graph=True),
        # One 7B draft tree: depth 6, width 8, vocabulary 65536, 64 nodes kept.
        dict(name="draft_7b", kind="draft", depth=6, width=8, V=65536, n_nodes=64, cfg=False, temperature=1.0,
             graph=True),
        # A LlamaGen-class wide draft under guidance: width 39, vocabulary 16384, 256 nodes kept.
        dict(name="draft_wide_guided", kind="draft", depth=5, width=39, V=16384, n_nodes=256, cfg=True,
             temperature=1.0, graph=False),
        # The verify phase of a small greedy step (26 nodes, vocabulary 16384, one layer's cache).
        dict(name="verify_greedy", kind="verify", mode="greedy", nodes="26", accept=2, V=16384, cfg=False,
             temperature=1.0, layers=1, Hkv=8, D=64, kv="512", lmax=576, max_path=10, graph=False),
        # The verify phase of a 7B step at T = 1 with a sampled draft (Eq. 1 with its residuals).  No drafted
        # token is kept, as in most steps at T = 1 (the paper's mean there is 1.1 tokens a step).
        dict(name="verify_spec_7b", kind="verify", mode="spec", nodes="64", accept=0, V=65536, cfg=False,
             temperature=1.0, layers=32, Hkv=32, D=128, kv="2400", lmax=2464, max_path=10, graph=False),
        # The verify phase of eight guided LlamaGen images, sampled, with top-k drafts.
        dict(name="verify_det_guided8", kind="verify", mode="spec_det", nodes="64,64,61,64,33,64,17,64", accept=0,
             V=16384, cfg=True, temperature=0.9, layers=36, Hkv=20, D=64, kv="696,120,388,512,244,640,301,575",
             lmax=760, max_path=10, graph=False),
        # The benchmark's whole step: draft, 32 layers of attention, greedy verify, commit.
        dict(name="step_7b", kind="step", layers=32, H=32, Hkv=32, D=128, V=65536, kv="2400", depth="6", width="8",
             max_nodes=64, accept=3, mode="greedy"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["attn"] * 5 + ["draft"] * 2 + ["verify"] * 3 + ["step"])
    if kind == "attn":
        D = rng.choice([64, 128])
        H = rng.choice([8, 20, 32])
        Hkv = rng.choice([H, H, H // 4])
        nb = rng.choice([1, 1, 2, 3, 4, 6, 8])
        if rng.random() < 0.15:  # the prompt: a chain of tokens before any cache
            nodes = [_log_int(rng, 2, 64)] * nb
            kv, chain, cap = [0] * nb, True, 64
        else:
            cap = rng.choice([26, 64, 64, 64, 128, 256])
            nodes = [rng.randint(max(1, cap // 8), cap) for _ in range(nb)]
            kv, chain = [_log_int(rng, 100, 6000) for _ in range(nb)], False
            if rng.random() < 0.2:
                cap = 256
        per_layer = sum(4 * (L + n) * Hkv * D + 4 * n * H * D for L, n in zip(kv, nodes))
        layers = max(1, min(rng.choice([1, 8, 32]), int(6e8 // per_layer)))
        return dict(kind=kind, layers=layers, kv=_text(kv), nodes=_text(nodes), max_nodes=cap, H=H, Hkv=Hkv, D=D,
                    lmax=max(kv) + cap + rng.randint(0, 64), chain=chain, lse=rng.random() < 0.3, graph=layers > 1)
    if kind == "draft":
        width = rng.choice([rng.randint(1, 8), rng.randint(4, 13), rng.randint(4, 39)])
        depth = rng.randint(1, 9)
        pool = width + (depth - 1) * width * width
        return dict(kind=kind, depth=depth, width=width, V=_log_int(rng, 4096, 65536),
                    n_nodes=min(pool + 1, rng.choice([26, 64, 64, 256])), cfg=rng.random() < 0.4,
                    temperature=rng.choice([1.0, 1.0, 0.8]), graph=rng.random() < 0.5)
    if kind == "verify":
        nb = rng.choice([1, 1, 2, 4, 8])
        cap = rng.choice([26, 64, 64, 256])
        nodes = [rng.randint(max(2, cap // 4), cap) for _ in range(nb)]
        layers, Hkv, D = rng.choice([(1, 8, 64), (36, 20, 64), (32, 32, 128)])
        kv = [_log_int(rng, 100, 2400 if nb == 1 else 600) for _ in range(nb)]
        mode = rng.choice(["greedy", "spec", "spec_det"])
        return dict(kind=kind, mode=mode, nodes=_text(nodes), accept=rng.randint(0, 5) if mode == "greedy" else 0,
                    V=_log_int(rng, 4096, 65536 if cap < 256 else 16384), cfg=rng.random() < 0.3,
                    temperature=1.0 if mode == "greedy" else rng.choice([1.0, 0.9]), layers=layers, Hkv=Hkv, D=D,
                    kv=_text(kv), lmax=max(kv) + cap, max_path=10, graph=False)
    layers, H, D = rng.choice([(12, 20, 64), (8, 32, 128)])
    nb = rng.choice([1, 2, 4])
    return dict(kind="step", layers=layers, H=H, Hkv=H, D=D, V=_log_int(rng, 4096, 65536) // 4 * 4,
                kv=_text(_log_int(rng, 120, 2400) for _ in range(nb)), depth=_text(rng.randint(2, 9) for _ in range(nb)),
                width=_text(rng.randint(2, 13) for _ in range(nb)), max_nodes=64, accept=rng.randint(0, 2),
                mode="greedy")


# ------------------------------------------------------------------ inputs

def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _bf16(g, *shape):
    return torch.randn(shape, generator=g, device=DEV, dtype=torch.float32).to(torch.bfloat16) if len(shape) < 5 else \
        torch.stack([_bf16(g, *shape[1:]) for _ in range(shape[0])])


def _rows(g, n, V, std=3.0):
    """[n, V] fp32 logits ~ N(0, std^2); the row stride is a multiple of 4 floats, as the ABI asks."""
    ld = (V + 3) // 4 * 4
    return (torch.randn((n, ld), generator=g, device=DEV) * std)[:, :V]


def _i32(x):
    return torch.as_tensor(list(x), dtype=torch.int32, device=DEV)


def _offsets(sizes):
    offs = [0]
    for n in sizes:
        offs.append(offs[-1] + n)
    return offs


def _tree_parents(sizes, seed, chain=False):
    """Parents of every tree, one list each (layered random trees, as drafts are)."""
    trees = []
    for b, n in enumerate(sizes):
        if chain:
            trees.append(synth.chain_tree(n).tolist())
        else:
            depth, kids = (6, 8) if n <= 64 else (9, 39)
            trees.append(synth.random_tree(n, int(seed) % (1 << 31), f"tree{b}", depth, kids).tolist())
    return trees


def _grown_parents(sizes, seed):
    """Parents of every tree, grown like a draft: layers of a fixed width, the root's children first."""
    trees = []
    for b, n in enumerate(sizes):
        pick, width = synth.rng(int(seed) % (1 << 31), f"grown{b}"), 4 if n <= 32 else 10 if n <= 64 else 39
        t, prev = [-1], [0]
        while len(t) < n:
            size = min(width, n - len(t))
            layer = list(range(len(t), len(t) + size))
            t += sorted(int(x) for x in pick.choice(prev, size=size))
            prev = layer
        trees.append(t)
    return trees


def _attn_inputs(case, seed):
    g = _gen(seed)
    L, H, Hkv, D, lmax = (case[k] for k in ("layers", "H", "Hkv", "D", "lmax"))
    kv, nodes = _ints(case["kv"]), _ints(case["nodes"])
    ntot = sum(nodes)
    return dict(kv=kv, nodes=nodes, trees=_tree_parents(nodes, seed, case["chain"]), q=_bf16(g, L, ntot, H, D),
                kt=_bf16(g, L, ntot, Hkv, D), vt=_bf16(g, L, ntot, Hkv, D), kc=_bf16(g, L, len(kv), Hkv, lmax, D),
                vc=_bf16(g, L, len(kv), Hkv, lmax, D))


def _draft_inputs(case, seed):
    g = _gen(seed)
    d, k, V = case["depth"], case["width"], case["V"]
    rows = [_rows(g, 1 if i == 0 else k, V) for i in range(d)]
    # the unconditional branch: the same image context without the text, so close to the conditional one
    rows_u = [r + _rows(g, r.shape[0], V, 0.5) for r in rows] if case["cfg"] else None
    if rows_u is not None:
        rows_u = [_pad(r) for r in rows_u]
    return dict(rows=rows, rows_u=rows_u, root=_i32([int(seed) % V]))


def _pad(rows):
    """The same rows with a row stride that is a multiple of 4 floats."""
    n, V = rows.shape
    out = torch.zeros((n, (V + 3) // 4 * 4), dtype=rows.dtype, device=rows.device)
    out[:, :V] = rows
    return out[:, :V]


def _plant(row, token, p, row_u=None):
    """Gives `token` probability p under softmax(row), for rows that the target is sure about."""
    v = torch.logsumexp(row.double(), 0) + math.log(p / (1 - p))
    row[token] = v.float()
    if row_u is not None:
        row_u[token] = v.float()


def _verify_inputs(case, seed):
    """Trees whose children are the draft rows' best tokens and targets close to the draft.  Greedy: on one root path
    per tree (of `accept` drafted nodes, where the tree is that deep) the target prefers the drafted token.  Sampling:
    the target has no use for any drafted token (probability about e^-60), so every child is tried and rejected."""
    g = _gen(seed)
    V, nodes, kv = case["V"], _ints(case["nodes"]), _ints(case["kv"])
    L, Hkv, D, lmax = (case[k] for k in ("layers", "Hkv", "D", "lmax"))
    trees = _grown_parents(nodes, seed)
    ntot, offs = sum(nodes), _offsets(nodes)
    kids_of = [[[i for i, p in enumerate(t) if p == v] for v in range(len(t))] for t in trees]
    most = max(len(k) for tree in kids_of for k in tree)
    inner = [(b, v) for b, tree in enumerate(kids_of) for v, k in enumerate(tree) if k]
    draft = _rows(g, max(1, len(inner)), V)
    best = torch.topk(draft, max(1, most), dim=1).indices.cpu().tolist()
    tokens, draft_row = [0] * ntot, [-1] * ntot
    target = _rows(g, ntot, V)
    index = [offs[b] + v for b, v in inner]
    if inner:
        target[torch.as_tensor(index, device=DEV)] = draft + _rows(g, len(inner), V, 0.5)
    for r, (b, v) in enumerate(inner):
        draft_row[offs[b] + v] = r
        for j, c in enumerate(kids_of[b][v]):
            tokens[offs[b] + c] = best[r][j]
    target_u = _pad(target + _rows(g, ntot, V, 0.5)) if case["cfg"] else None
    draft_u = _pad(draft + _rows(g, draft.shape[0], V, 0.5)) if case["cfg"] else None
    if case["mode"] != "greedy" and inner:
        rows, cols = zip(*((offs[b] + t[i], tokens[offs[b] + i]) for b, t in enumerate(trees) for i in range(1, len(t))))
        low = target.max() - 60.0
        for t in (target, target_u) if case["cfg"] else (target,):
            t[list(rows), list(cols)] = low
    for b, t in enumerate(trees):
        depth = [0] * len(t)
        for i in range(1, len(t)):
            depth[i] = depth[t[i]] + 1
        node = max(range(len(t)), key=lambda i: (min(depth[i], case["accept"]), -i))
        while case["mode"] == "greedy" and node > 0:
            row = offs[b] + t[node]
            _plant(target[row], tokens[offs[b] + node], 0.85, None if target_u is None else target_u[row])
            node = t[node]
    return dict(nodes=nodes, parents=_i32(p for t in trees for p in t), offs=_i32(offs), tokens=_i32(tokens),
                draft_row=_i32(draft_row), target=target, target_u=target_u, draft=draft, draft_u=draft_u,
                ua=torch.rand(ntot, generator=g, device=DEV).clamp_min(2.0 ** -24), us=torch.rand(ntot, generator=g, device=DEV),
                kv=_i32(kv), kt=_bf16(g, L, ntot, Hkv, D), vt=_bf16(g, L, ntot, Hkv, D),
                kc=_bf16(g, L, len(kv), Hkv, lmax, D), vc=_bf16(g, L, len(kv), Hkv, lmax, D))


def _step_shape(case):
    return StepShape(layers=case["layers"], H=case["H"], Hkv=case["Hkv"], D=case["D"], V=case["V"],
                     kv_len=_ints(case["kv"]), depth=_ints(case["depth"]), width=_ints(case["width"]),
                     max_nodes=case["max_nodes"], mode=MODES[case["mode"]])


def _step_inputs(step, case, seed):
    g = _gen(seed)
    for name in ("q", "k_tree", "v_tree", "k_cache", "v_cache"):
        t = getattr(step, name)
        for layer in range(t.shape[0]):
            t[layer] = _bf16(g, *t.shape[1:])
    step.target.copy_(_rows(g, step.ntot, case["V"]))
    for rows in step.draft_rows:
        rows.copy_(torch.randn(rows.shape, generator=g, device=DEV) * 3.0)
    step.root_token.copy_(_i32((int(seed) + b) % case["V"] for b in range(len(step.n))))


# ------------------------------------------------------------------ passes

def _attn_state(case, seed):
    i = _attn_inputs(case, seed)
    L, H, Hkv, D = (case[k] for k in ("layers", "H", "Hkv", "D"))
    nb, ntot = len(i["kv"]), sum(i["nodes"])
    kv_len, offs = _i32(i["kv"]), _i32(_offsets(i["nodes"]))
    parents = _i32(p for t in i["trees"] for p in t)
    out = torch.zeros((L, ntot, H, D), dtype=torch.bfloat16, device=DEV)
    lse = torch.zeros((L, ntot, H), dtype=torch.float32, device=DEV) if case["lse"] else None
    ws = B.zeroed_workspace(B.adt_tree_attn_workspace_size(nb, H, D, case["max_nodes"], case["lmax"]))
    q, kc, vc, kt, vt = i["q"], i["kc"], i["vc"], i["kt"], i["vt"]

    def passes():
        for la in range(L):
            B.adt_tree_attn(q[la], kc[la], vc[la], kv_len, kt[la], vt[la], parents, offs, B=nb, H=H, Hkv=Hkv, D=D,
                            max_nodes=case["max_nodes"], max_kv=case["lmax"], softmax_scale=D ** -0.5, out=out[la],
                            lse=None if lse is None else lse[la], workspace=ws)

    return passes, dict(out=out) if lse is None else dict(out=out, lse=lse)


def _draft_state(case, seed):
    i = _draft_inputs(case, seed)
    d, k, V, n = (case[x] for x in ("depth", "width", "V", "n_nodes"))
    C = k + (d - 1) * k * k
    i32, f32 = dict(dtype=torch.int32, device=DEV), dict(dtype=torch.float32, device=DEV)
    pool = dict(child_token=torch.zeros(C, **i32), child_logp=torch.zeros(C, **f32), child_score=torch.zeros(C, **f32),
                child_parent=torch.zeros(C, **i32))
    tree = {x: torch.zeros(n, **i32) for x in ("tokens", "parents", "cand_index", "depth")}
    front = [(torch.zeros(1, **f32), torch.full((1,), -1, **i32))] + \
        [(torch.zeros(k, **f32), torch.zeros(k, **i32)) for _ in range(d - 1)]
    keep = torch.zeros(k, **i32)
    ws, ws_r = B.zeroed_workspace(B.adt_tree_expand_workspace_size(k, V, k)), \
        B.zeroed_workspace(B.adt_tree_rerank_workspace_size(C))

    def passes():
        base = 0
        for la in range(d):
            F = 1 if la == 0 else k
            nxt = front[la + 1] if la + 1 < d else (None, None)
            args = dict(F=F, V=V, k_child=k, k_keep=k, temperature=case["temperature"], child_id_base=base,
                        keep_idx=keep if la + 1 < d else None, next_score=nxt[0], next_id=nxt[1], workspace=ws,
                        **{x: t[base:base + F * k] for x, t in pool.items()})
            if case["cfg"]:
                B.adt_tree_expand_cfg(i["rows"][la], i["rows_u"][la], *front[la], cfg_scale=3.0, **args)
            else:
                B.adt_tree_expand(i["rows"][la], *front[la], **args)
            base += F * k
        B.adt_tree_rerank(pool["child_token"], pool["child_score"], pool["child_parent"], C, i["root"], n,
                          workspace=ws_r, **tree)

    return passes, dict(pool=pool, tree=tree)


def _verify_state(case, seed):
    i = _verify_inputs(case, seed)
    nb, V, mp = len(i["nodes"]), case["V"], case["max_path"]
    i32 = dict(dtype=torch.int32, device=DEV)
    path, alen, bonus, kv_out = torch.zeros((nb, mp), **i32), torch.zeros(nb, **i32), torch.zeros(nb, **i32), \
        torch.zeros(nb, **i32)
    mode = MODES[case["mode"]]
    args = dict(B=nb, V=V, max_nodes=max(i["nodes"]), mode=mode, u_accept=i["ua"], u_sample=i["us"],
                temperature=case["temperature"], path=path, max_path=mp, accept_len=alen, bonus_token=bonus)
    spec = mode == B.ACCEPT_SPEC
    if spec:
        args["draft_row"] = i["draft_row"]
    kc, vc, kt, vt = i["kc"], i["vc"], i["kt"], i["vt"]

    def passes():
        if case["cfg"]:
            B.adt_tree_accept_cfg(i["target"], i["target_u"], i["draft"] if spec else None,
                                  i["draft_u"] if spec else None, i["tokens"], i["parents"], i["offs"], cfg_scale=3.0,
                                  **args)
        else:
            B.adt_tree_accept(i["target"], i["draft"] if spec else None, i["tokens"], i["parents"], i["offs"], **args)
        B.adt_kv_compact(kc, vc, i["kv"], kv_out, kt, vt, i["offs"], path, mp, alen, B=nb, Hkv=case["Hkv"], D=case["D"],
                         num_layers=case["layers"], max_kv=case["lmax"], cache_layer_stride=kc.stride(0),
                         cache_stride_b=kc.stride(1), cache_stride_h=kc.stride(2), tree_layer_stride=kt.stride(0))

    return passes, dict(path=path, accept_len=alen, bonus=bonus, kv_len=kv_out, k_cache=kc, v_cache=vc)


def _step_state(case, seed):
    step = TreeVerifyStep(_step_shape(case), keep_layer_outputs=True)
    _step_inputs(step, case, seed)
    # a target that agrees with the draft on one root path of `accept` nodes per tree
    step.launch_draft()
    tokens, parents = step.tokens.cpu().tolist(), step.parents.cpu().tolist()
    for b, lo in enumerate(_offsets(step.n)[:-1]):
        t = parents[lo:lo + step.n[b]]
        depth = [0] * len(t)
        for i in range(1, len(t)):
            depth[i] = depth[t[i]] + 1
        node = max(range(len(t)), key=lambda i: (min(depth[i], case["accept"]), -i))
        while node > 0:
            _plant(step.target[lo + t[node]], tokens[lo + node], 0.85)
            node = t[node]
    outs = dict(tokens=step.tokens, parents=step.parents, depth=step.node_depth, attn=step.attn_out, path=step.path,
                accept_len=step.accept_len, bonus=step.bonus, kv_len=step.kv_len_out, k_cache=step.k_cache,
                v_cache=step.v_cache)
    return step.launch, outs


def prepare(case, seed):
    make = dict(attn=_attn_state, draft=_draft_state, verify=_verify_state, step=_step_state)[case["kind"]]
    passes, outs = make(case, seed)
    if case.get("graph", case["kind"] == "step"):
        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side):
            passes()
        torch.cuda.current_stream().wait_stream(side)
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            passes()
        return dict(run=graph.replay, outs=outs, keep=(graph, passes))
    return dict(run=passes, outs=outs)


def run(state):
    state["run"]()
    return state["outs"]


# ------------------------------------------------------------------ accounting

def _attn_bytes(kv, nodes, H, Hkv, D):
    return sum(4 * (L + n) * Hkv * D + 4 * n * H * D for L, n in zip(kv, nodes))


def _attn_flops(kv, nodes, H, D):
    return sum(4 * n * (L + n) * H * D for L, n in zip(kv, nodes))


def work(case):
    if case["kind"] == "attn":
        kv, nodes = _ints(case["kv"]), _ints(case["nodes"])
        return dict(bytes=case["layers"] * _attn_bytes(kv, nodes, case["H"], case["Hkv"], case["D"]),
                    flops=case["layers"] * _attn_flops(kv, nodes, case["H"], case["D"]))
    if case["kind"] == "draft":
        k, d = case["width"], case["depth"]
        rows, pool = 1 + (d - 1) * k, k + (d - 1) * k * k
        return dict(bytes=rows * case["V"] * 4 * (2 if case["cfg"] else 1) + 16 * pool + 16 * case["n_nodes"],
                    flops=3 * rows * case["V"])
    if case["kind"] == "verify":
        nb = len(_ints(case["nodes"]))
        rows = nb * (case["accept"] + 1)  # the rows of the planted path
        per_row = case["V"] * 4 * (2 if case["cfg"] else 1) * (2 if case["mode"] == "spec" else 1)
        commit = rows * case["layers"] * case["Hkv"] * case["D"] * 2 * 2 * 2
        return dict(bytes=rows * per_row + commit, flops=3 * rows * per_row / 4)
    kv, d, k = _ints(case["kv"]), _ints(case["depth"]), _ints(case["width"])
    pools = [w + (x - 1) * w * w for x, w in zip(d, k)]
    nodes = [min(case["max_nodes"], c + 1) for c in pools]
    rows = sum(1 + (x - 1) * w for x, w in zip(d, k)) + len(kv) * (case["accept"] + 1)
    commit = len(kv) * (case["accept"] + 1) * case["layers"] * case["Hkv"] * case["D"] * 8
    return dict(bytes=case["layers"] * _attn_bytes(kv, nodes, case["H"], case["Hkv"], case["D"]) + rows * case["V"] * 4
                + commit, flops=case["layers"] * _attn_flops(kv, nodes, case["H"], case["D"]) + 3 * rows * case["V"])


def tolerance(case):
    if case["kind"] in ("attn", "step"):
        # bf16 probabilities and a bf16 result, each rounded by up to 2^-9: 0.0024 from the fp64 result, measured
        return {"rel": 1e-2, "max": 0.05}
    if case["kind"] == "draft":
        # log-probabilities and scores in fp32 (4.6e-8 from fp64, measured); token ids and trees are the same
        return {"rel": 2e-7, "max": 2e-6}
    return "exact"


# ------------------------------------------------------------------ the same in 64 bits

def _attn_exact(q, kc, vc, kt, vt, trees, kv, H, Hkv, D):
    """One layer in fp64: (out [ntot, H, D], lse [ntot, H])."""
    outs, lses, lo = [], [], 0
    for b, t in enumerate(trees):
        n, L = len(t), kv[b]
        vis = torch.zeros((n, n), dtype=torch.bool)
        for i, p in enumerate(t):
            if p >= 0:
                vis[i] = vis[p]
            vis[i, i] = True
        bias = torch.zeros((n, L + n), dtype=torch.float64, device=DEV)
        bias[:, L:].masked_fill_(~vis.to(DEV), -math.inf)
        rep = H // Hkv
        K = torch.cat([kc[b, :, :L], kt[lo:lo + n].transpose(0, 1)], 1).double().repeat_interleave(rep, 0)
        V = torch.cat([vc[b, :, :L], vt[lo:lo + n].transpose(0, 1)], 1).double().repeat_interleave(rep, 0)
        s = q[lo:lo + n].transpose(0, 1).double() @ K.transpose(1, 2) * D ** -0.5 + bias
        lse = torch.logsumexp(s, -1)
        outs.append((torch.exp(s - lse[..., None]) @ V).transpose(0, 1))
        lses.append(lse.transpose(0, 1))
        lo += n
    return torch.cat(outs), torch.cat(lses)


def _draft_exact(rows, rows_u, width, temperature, n_nodes):
    """Draft growth with fp64 log-probabilities: pool log-probabilities and scores, and the kept tree's parents."""
    logp, score, par = [], [], []
    fscore, fid, base = torch.zeros(1, dtype=torch.float64, device=DEV), [-1], 0
    for la, r in enumerate(rows):
        x = r.float()
        if rows_u is not None:  # the guided logits, each operation rounded to fp32
            x = rows_u[la] + 3.0 * (x - rows_u[la])
        if temperature != 1.0:
            x = x / torch.tensor(temperature, dtype=torch.float32, device=DEV)
        top = torch.sort(x, dim=1, descending=True, stable=True).values[:, :width]
        lp = top.double() - torch.logsumexp(x.double(), 1, keepdim=True)
        sc = (fscore[:, None] + lp).reshape(-1)
        logp.append(lp.reshape(-1))
        score.append(sc)
        par += [fid[c // width] for c in range(sc.numel())]
        keep = torch.sort(sc, descending=True, stable=True).indices[:width]
        fscore, fid = sc[keep], [base + c for c in keep.cpu().tolist()]
        base += sc.numel()
    logp, score = torch.cat(logp), torch.cat(score)
    chosen = sorted(torch.sort(score, descending=True, stable=True).indices[:n_nodes - 1].cpu().tolist())
    node = {c: j + 1 for j, c in enumerate(chosen)}
    return logp, score, [-1] + [0 if par[c] < 0 else node[par[c]] for c in chosen]


def exact(case, seed):
    if case["kind"] == "attn":
        i = _attn_inputs(case, seed)
        got = [_attn_exact(i["q"][la], i["kc"][la], i["vc"][la], i["kt"][la], i["vt"][la], i["trees"], i["kv"],
                           case["H"], case["Hkv"], case["D"]) for la in range(case["layers"])]
        out = torch.stack([o for o, _ in got])
        return dict(out=out, lse=torch.stack([x for _, x in got])) if case["lse"] else dict(out=out)
    if case["kind"] == "draft":
        i = _draft_inputs(case, seed)
        logp, score, _ = _draft_exact(i["rows"], i["rows_u"], case["width"], case["temperature"], case["n_nodes"])
        return dict(pool=dict(child_token=None, child_logp=logp, child_score=score, child_parent=None), tree=None)
    if case["kind"] == "step":
        step = TreeVerifyStep(_step_shape(case), keep_layer_outputs=True)  # its buffers hold the inputs
        _step_inputs(step, case, seed)
        kv, d, k = _ints(case["kv"]), _ints(case["depth"]), _ints(case["width"])
        trees = [_draft_exact([r[x, :1 if x == 0 else k[b]] for x in range(d[b])], None, k[b], 1.0, step.n[b])[2]
                 for b, r in enumerate(step.draft_rows)]
        out = torch.stack([_attn_exact(step.q[la], step.k_cache[la], step.v_cache[la], step.k_tree[la],
                                       step.v_tree[la], trees, kv, case["H"], case["Hkv"], case["D"])[0]
                           for la in range(case["layers"])])
        none = {x: None for x in ("tokens", "parents", "depth", "path", "accept_len", "bonus", "kv_len", "k_cache",
                                  "v_cache")}
        return dict(attn=out, **none)
    return None  # a walk's decisions are whole numbers, and the commit copies bytes
