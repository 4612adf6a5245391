"""Sampling walks that accept drafted nodes, repeated.  The CTAs of a tree's
cluster read each other's slices of p and q while the children are tried, and
an accepted child's row overwrites those slices: without a cluster barrier
between the two a slower CTA reads the next row's values and decides
otherwise than its peers.  Every one of many back-to-back walks has to give
the oracle's path, length and bonus token."""
import numpy as np
import pytest
import torch

import oracle
from gpu_cases import ensure_built, f32, f32_rows, i32
from paper_2512_21857_gb300 import binding as B
from paper_2512_21857_gb300 import synth
from test_parity_accept_compact import ACCEPT_MARGIN, SAMPLE_MARGIN, compare, make_rows

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", [B.ACCEPT_SPEC, B.ACCEPT_SPEC_DET])
def test_accepting_walks_repeat(mode):
    ensure_built()
    sizes, V, reps, max_path = [64, 33, 50, 17, 64, 61, 26, 40], 16384, 400, 16
    for seed in range(40, 60):
        tb = synth.tree_batch(sizes, V, seed, max_depth=8, max_children=6)
        target, draft = make_rows(tb, V, seed, 0.3)
        ua = synth.uniforms(len(tb.tokens), seed, "ua")
        us = synth.uniforms(len(tb.tokens), seed, "us")
        res = oracle.tree_accept(target, draft, tb.tokens, tb.parents, tb.node_offsets, mode, ua, us)
        if res["accept_margin"] > ACCEPT_MARGIN and res["sample_margin"] > SAMPLE_MARGIN:
            break
    assert sum(res["accept_len"]) >= 8
    args = (f32_rows(target), f32_rows(draft) if mode == B.ACCEPT_SPEC else None, i32(tb.tokens), i32(tb.parents),
            i32(tb.node_offsets))
    ua_d, us_d, nb = f32(ua), f32(us), len(sizes)
    path = torch.zeros((reps, nb, max_path), dtype=torch.int32, device="cuda")
    alen, bonus = (torch.zeros((reps, nb), dtype=torch.int32, device="cuda") for _ in range(2))
    for r in range(reps):
        B.adt_tree_accept(*args, B=nb, V=V, max_nodes=64, mode=mode, u_accept=ua_d, u_sample=us_d, path=path[r],
                          max_path=max_path, accept_len=alen[r], bonus_token=bonus[r])
    torch.cuda.synchronize()
    compare(tb, res, path[0].cpu().numpy(), alen[0].cpu().numpy(), bonus[0].cpu().numpy())
    for t in (path, alen, bonus):
        assert torch.equal(t, t[:1].expand_as(t))
