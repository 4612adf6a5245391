"""Sampling walks at nodes with many children: more than a batch (64) of them,
tokens that occur twice, tokens without probability and outside the
vocabulary, walks that reject all, a few or none of them, with double-float
and fp32 slices.  Paths, lengths and bonus tokens match the oracle bit for
bit wherever its decision margins allow (1e-9; fp32 slices: 1e-5)."""
import numpy as np
import pytest

import oracle
from gpu_cases import ensure_built, run_accept_gpu
from paper_2512_21857_gb300 import binding as B
from paper_2512_21857_gb300 import synth
from test_parity_accept_compact import compare, make_rows

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    ensure_built()


def _star(kids, V, seed, low, sigma=0.5):
    """A root with `kids` children, each of them with two; targets close to
    the draft, but without use for the children listed in `low`."""
    parents = [-1] + [0] * kids + sorted(list(range(1, kids + 1)) * 2)
    tb = synth.TreeBatch(np.asarray(parents, np.int32), synth.tree_tokens(np.asarray(parents, np.int32), V, seed),
                         np.asarray([0, len(parents)], np.int32))
    draft = synth.f32_normal((len(parents), V), seed, "draft", std=2.0)
    target = (draft + synth.f32_normal((len(parents), V), seed, "noise", std=sigma)).astype(np.float32)
    for c in low:
        target[0, tb.tokens[c]] = -60.0
    return tb, target, draft


def _check(tb, target, draft, mode, seed, margin=1e-9, T=1.0):
    n = len(tb.tokens)
    ua, us = synth.uniforms(n, seed, "ua"), synth.uniforms(n, seed, "us")
    ua[ua == 0] = 0.5
    res = oracle.tree_accept(target, draft, tb.tokens, tb.parents, tb.node_offsets, mode, ua, us, T)
    if res["min_margin"] < margin:
        return None
    compare(tb, res, *run_accept_gpu(target, draft if mode == B.ACCEPT_SPEC else None, tb, mode, ua, us, T))
    return int(res["accept_len"][0])


@pytest.mark.parametrize("mode", [B.ACCEPT_SPEC, B.ACCEPT_SPEC_DET])
@pytest.mark.parametrize("kids", [1, 31, 33, 64, 65, 150])
def test_many_children(kids, mode):
    got = []
    for seed in range(6):
        tb, target, draft = _star(kids, 5003, 100 * kids + seed, range(1, kids + 1 - (seed % 3)))
        got.append(_check(tb, target, draft, mode, seed))
    assert sum(g is not None for g in got) >= 5
    assert 0 in got


@pytest.mark.parametrize("mode", [B.ACCEPT_SPEC, B.ACCEPT_SPEC_DET])
@pytest.mark.parametrize("kids", [6, 40, 100])
def test_repeated_tokens(kids, mode):
    checked = 0
    for seed in range(6):
        tb, target, draft = _star(kids, 4096, 7 * kids + seed, range(1, kids, 2))
        g = np.random.default_rng(seed)
        for c in range(2, kids + 1, 3):
            tb.tokens[c] = tb.tokens[int(g.integers(1, c))]
        checked += _check(tb, target, draft, mode, seed, T=0.8) is not None
    assert checked >= 5


def test_a_draft_equal_to_its_target_keeps_p():
    """Rejecting a token of zero probability under p = q leaves no residual
    mass: p stays as it is, the draft only loses the token."""
    for kids in (3, 70):
        tb, target, draft = _star(kids, 4096, kids, [], sigma=0.0)
        for c in range(1, kids):
            target[0, tb.tokens[c]] = draft[0, tb.tokens[c]] = -3000.0
        assert _check(tb, target, draft, B.ACCEPT_SPEC, 1) is not None


def test_a_token_outside_the_vocabulary_is_skipped():
    """As if its probability were zero (which a deterministic draft's
    rejection does not change anything by), and flagged."""
    tb, target, draft = _star(20, 4096, 3, range(1, 19))
    target[0, tb.tokens[2]] = -3000.0
    n = len(tb.tokens)
    ua, us = synth.uniforms(n, 5, "ua"), synth.uniforms(n, 5, "us")
    res = oracle.tree_accept(target, None, tb.tokens, tb.parents, tb.node_offsets, B.ACCEPT_SPEC_DET, ua, us)
    assert res["min_margin"] > 1e-9
    tb.tokens[2] = 4096
    B.adt_get_device_error()
    compare(tb, res, *run_accept_gpu(target, None, tb, B.ACCEPT_SPEC_DET, ua, us))
    assert B.adt_get_device_error() == B.DEVERR_BAD_INDEX


@pytest.mark.parametrize("V", [40000, 262144])
def test_cluster_sizes_and_fp32_slices(V):
    """16 CTAs for one tree; past about 210000 entries the slices are fp32."""
    checked = 0
    for seed in range(4):
        tb, target, draft = _star(12, V, V + seed, range(1, 12))
        checked += _check(tb, target, draft, B.ACCEPT_SPEC, seed, margin=1e-9 if V < 200000 else 1e-5) is not None
    assert checked >= 2


@pytest.mark.parametrize("trees,V", [(16, 32768), (20, 4099), (40, 4096), (77, 16384), (17, 40000)])
def test_many_trees(trees, V):
    """SPEC with 4, 4, 2, 2 and 8 CTAs a tree, in one wave and in two."""
    for seed in range(V, V + 20):
        tb = synth.tree_batch([1 + (5 * i) % 13 for i in range(trees)], V, seed, max_depth=4, max_children=6)
        target, draft = make_rows(tb, V, seed, 0.3)
        n = len(tb.tokens)
        ua, us = synth.uniforms(n, seed, "ua"), synth.uniforms(n, seed, "us")
        res = oracle.tree_accept(target, draft, tb.tokens, tb.parents, tb.node_offsets, B.ACCEPT_SPEC, ua, us)
        if res["min_margin"] > 1e-9:
            break
    assert res["min_margin"] > 1e-9
    compare(tb, res, *run_accept_gpu(target, draft, tb, B.ACCEPT_SPEC, ua, us))
