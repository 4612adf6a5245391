"""Wide drafts: the expansion's selections past 8 children a row (64 group
maxima bound the keys that are ranked, radix selection where too many reach
the bound), its split of a row over fewer CTAs when there are many rows, and
the rerank of large pools (score bins, then the threshold bin ranked)."""
import numpy as np
import pytest
import torch

import oracle
from gpu_cases import ensure_built, f32, i32
from paper_2512_21857_gb300 import binding as B
from paper_2512_21857_gb300 import synth
from test_parity_cfg import run_expand_cfg
from test_parity_expand_rerank import _random_pool, check_expand, run_expand

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    ensure_built()


@pytest.mark.parametrize("F,V,k,keep", [
    (8, 65536, 8, 8), (9, 65536, 8, 8),      # 64 and 72 cross-row keys
    (8, 65536, 9, 9),                        # 72 keys in a row's lists
    (3, 16384, 32, 32), (3, 16384, 33, 33),  # warp maxima, half-warp maxima
    (20, 65536, 20, 20),                     # 6 CTAs a row
    (39, 65536, 39, 64),                     # 2 CTAs a row, a full tile each, 64 kept of 1521
    (16, 4100, 64, 64),                      # 1024 cross-row keys
    (130, 40000, 5, 100),                    # one CTA a row, two tiles; k_keep past 64
])
def test_expand_wide_matches_oracle(F, V, k, keep):
    logits = synth.f32_normal((F, V), F + V + k, "logits", std=3.0)
    fscore = synth.f32_normal((F,), F + V + k, "fs", std=1.0) - 2.0
    got, _ = run_expand(logits, fscore, None, k, keep, base=5)
    check_expand(got, oracle.tree_expand(logits, fscore, k, keep, child_id_base=5), keep)


@pytest.mark.parametrize("F,V,k", [(39, 65536, 39), (2, 4098, 8)])
def test_expand_guided_tiles_match_oracle(F, V, k):
    """Guidance halves the tile: two CTAs a row stage two tiles each at V = 65536."""
    V4 = (V + 3) // 4 * 4
    cond, uncond = (synth.f32_normal((F, V4), V + i, "l", std=3.0) for i in range(2))
    fscore = synth.f32_normal((F,), V, "fs", std=1.0)
    got = run_expand_cfg(cond, uncond, fscore, None, k, k)
    check_expand(got, oracle.tree_expand(oracle.cfg_logits(cond, uncond, 3.0), fscore, k, k), k)


def test_expand_cross_row_overflow_takes_the_radix_path():
    """63 of 64 children of every row far above the last one: the bound of
    the cross-row selection is a last child, and more keys reach it than the
    candidate buffer holds."""
    F, V, k = 40, 2048, 64
    logits = synth.f32_normal((F, V), 5, "logits", std=0.5)
    g = np.random.default_rng(5)
    for r in range(F):
        logits[r, g.choice(V, size=63, replace=False)] += np.float32(30.0)
    fscore = synth.f32_normal((F,), 6, "fs", std=0.1)
    got, _ = run_expand(logits, fscore, None, k, 64)
    check_expand(got, oracle.tree_expand(logits, fscore, k, 64), 64)


@pytest.mark.parametrize("n_top", [129, 1025])
def test_expand_ties_past_the_direct_ranking(n_top):
    """n_top copies of the largest value in one CTA's share, k = 40: ranked
    after a second bound (129), or past the candidate buffer (1025)."""
    V, F, k = 65536, 2, 40
    g = np.random.default_rng(n_top)
    logits = g.normal(0.0, 1.0, size=(F, V)).astype(np.float32)
    pos = np.sort(g.choice(8192, size=n_top, replace=False)) + 8192 * 3
    logits[0, pos] = np.float32(7.0)
    fscore = np.array([-1.0, -0.25], np.float32)
    got, _ = run_expand(logits, fscore, None, k, k)
    assert got["child_token"][:k].tolist() == pos[:k].tolist()
    check_expand(got, oracle.tree_expand(logits, fscore, k, k), k)


def _rerank(tok, sc, par, n):
    C = len(tok)
    res = {x: torch.empty(n, dtype=torch.int32, device="cuda") for x in ("tokens", "parents", "cand_index", "depth")}
    ws = B.zeroed_workspace(B.adt_tree_rerank_workspace_size(C))
    B.adt_tree_rerank(i32(tok), f32(sc), i32(par), C, i32([7]), n, workspace=ws, **res)
    torch.cuda.synchronize()
    return {x: t.cpu().numpy() for x, t in res.items()}


@pytest.mark.parametrize("C,n", [(328, 64), (1024, 256), (1025, 2), (6123, 256), (8192, 4096), (8193, 257),
                                 (40000, 64), (65536, 4096)])
@pytest.mark.parametrize("scores", ["grown", "flat", "outlier", "masked"])
def test_rerank_large_pools(C, n, scores):
    """Scores as grown; all equal; all but one far away in one bin; the last third -inf."""
    tok, sc, par = _random_pool(C, seed=C + n)
    if scores == "flat":
        sc = np.full_like(sc, -3.0)
    elif scores == "outlier":
        sc = sc.copy()
        sc[0] = np.float32(1e30)
        par[:] = -1
    elif scores == "masked":
        sc, par = sc.copy(), np.full_like(par, -1)
        sc[2 * C // 3:] = -np.inf
    got, ref = _rerank(tok, sc, par, n), oracle.tree_rerank(tok, sc, par, 7, n)
    for key in got:
        assert np.array_equal(got[key], ref[key]), key


LOWEST = float(np.finfo(np.float32).min)


@pytest.mark.parametrize("C,n", [(40, 9), (128, 100), (129, 100), (200, 201), (328, 64), (1024, 256), (2048, 64),
                                 (2049, 2), (4096, 300), (6123, 257), (8193, 257), (40000, 700)])
@pytest.mark.parametrize("scores", ["decades", "lowest", "equal", "steps", "nan"])
def test_rerank_scores_that_crowd_a_bin(C, n, scores):
    """Scores whose range a few of them stretch, so that the rest share a bin,
    and equal ones: binned again, by value and then by index; pools ranked as
    they are (up to 128), selected whole, and too large for registers.  A NaN ranks
    first, one with its sign set last."""
    g = np.random.default_rng(C + n)
    sc = -g.exponential(size=C).astype(np.float32) * 3
    if scores == "decades":
        sc[g.choice(C, 30, replace=False)] = -10.0 ** np.arange(3, 33)
    elif scores == "lowest":
        sc[::5] = LOWEST
        sc[3::7] = -np.inf
        sc[1] = 3e38  # the range leaves fp32
    elif scores == "equal":
        sc[:] = -3.0
        sc[5] = 0.0
    elif scores == "steps":  # neighbouring values around the threshold, 300 of each
        sc = (np.float32(-1.0) - np.arange(C, dtype=np.float32) // 300 * np.float32(2.0 ** -23)).astype(np.float32)
        g.shuffle(sc)
        sc[0] = -1e20
    else:
        sc[g.choice(C, 9, replace=False)] = np.nan
        sc[2] = -np.float32(np.nan)
        sc[4] = np.inf
    got = _rerank(np.arange(C), sc, np.full(C, -1, np.int32), n)
    order = np.lexsort((np.arange(C), -np.where(np.isnan(sc), 0, sc.astype(np.float64)),
                        np.where(np.isnan(sc), np.where(np.signbit(sc), 1, -1), 0)))
    assert np.array_equal(got["cand_index"][1:], np.sort(order[:n - 1]))
    assert np.array_equal(got["tokens"][1:], got["cand_index"][1:])


@pytest.mark.parametrize("V,k", [(65536, 8), (16384, 39)])  # one row's CTAs: narrow and general instantiation
@pytest.mark.parametrize("mask", [LOWEST, -np.inf])
def test_expand_scores_outside_the_range_of_fp32(V, k, mask):
    """Rows with fewer than k unmasked logits and frontier scores at the ends
    of fp32: log-probabilities and scores are those of fp64 rounded once
    (-inf where the sum of two lowest values leaves the range)."""
    fscore = np.array([-1.0, LOWEST, -np.inf], np.float32)
    F = len(fscore)
    g = np.random.default_rng(k)
    logits = np.full((F, V), mask, np.float32)
    for r in range(F):
        logits[r, g.choice(V, size=k - 3, replace=False)] = g.normal(0.0, 2.0, size=k - 3)
    got, _ = run_expand(logits, fscore, None, k, k)
    with np.errstate(over="ignore"):
        for r in range(F):
            x = logits[r].astype(np.float64)
            m = x.max()
            order = np.argsort(-x, kind="stable")[:k]
            lp = x[order] - (m + np.log(np.exp(x - m).sum()))
            sl = slice(r * k, (r + 1) * k)
            assert got["child_token"][sl].tolist() == order.tolist()
            np.testing.assert_allclose(got["child_logp"][sl], lp.astype(np.float32), rtol=1e-6, atol=1e-6)
            np.testing.assert_allclose(got["child_score"][sl], (float(fscore[r]) + lp).astype(np.float32),
                                       rtol=1e-6, atol=1e-6)


@pytest.mark.parametrize("k", [8, 39])
@pytest.mark.parametrize("F,V", [(2, 2047), (2, 2048), (2, 2049), (3, 4097), (2, 65533), (2, 65536), (2, 65540),
                                 (16, 65536), (64, 16384), (77, 4096)])
def test_expand_share_in_registers(F, V, k):
    """Shares of one pair a thread to eight logits a thread, an odd logit at
    the end, and one logit less or more a share than registers are used for
    (2047; 8196 of 65540; 10924 in six CTAs), rows in pairs of CTAs and, one
    row more than pairs of SMs, in single ones; plain, divided by a
    temperature and guided."""
    logits = synth.f32_normal((F, V), V + k, "logits", std=3.0)
    fscore = synth.f32_normal((F,), V, "fs", std=1.0)
    keep = min(F * k, 64)
    for T in (1.0, 0.7):
        got, _ = run_expand(logits, fscore, None, k, keep, T=T)
        check_expand(got, oracle.tree_expand(logits, fscore, k, keep, temperature=T), keep)
    cond, uncond = (synth.f32_normal((F, V), V + i, "l", std=3.0) for i in range(2))
    got = run_expand_cfg(cond, uncond, fscore, None, k, keep)
    check_expand(got, oracle.tree_expand(oracle.cfg_logits(cond, uncond, 3.0), fscore, k, keep), keep)


@pytest.mark.parametrize("F,V,k", [
    (8, 65536, 8), (8, 16384, 39),  # shares in registers: narrow and general instantiation
    (8, 2047, 8), (8, 2047, 39),    # staged in shared memory
    (130, 40000, 9),                # two tiles
])
def test_expand_rows_of_any_magnitude(F, V, k):
    """Rows that lie wholly at fp32's lowest value, near it, around +-1e10 and
    2^20, beside ordinary ones: log-probabilities are those of fp64 (-ln V where all
    logits are equal), and such a row does not disturb the next frontier."""
    logits = synth.f32_normal((F, V), V + k, "logits", std=3.0)
    for r, level in ((1, LOWEST), (2, -3e38), (3, -1e10), (4, 1e10), (5, 3e38)):
        logits[r] = np.float32(level)
    logits[4, 5:V:7] = np.nextafter(np.float32(1e10), np.float32(0))  # 1024 below: no weight
    logits[0] += np.float32(2 ** 20 - 64)  # terms of either form
    logits[6] += np.float32(2 ** 20)
    fscore = synth.f32_normal((F,), V, "fs", std=1.0)
    got, _ = run_expand(logits, fscore, None, k, k)
    for r in range(F):
        x = logits[r].astype(np.float64)
        m = x.max()
        order = np.argsort(-x, kind="stable")[:k]
        lp = x[order] - m - np.log(np.exp(x - m).sum())
        sl = slice(r * k, (r + 1) * k)
        assert got["child_token"][sl].tolist() == order.tolist()
        np.testing.assert_allclose(got["child_logp"][sl], lp.astype(np.float32), rtol=1e-6, atol=1e-6)
        np.testing.assert_allclose(got["child_score"][sl], (float(fscore[r]) + lp).astype(np.float32), rtol=1e-6,
                                   atol=1e-6)
    assert got["keep_idx"].tolist() == np.argsort(-got["child_score"], kind="stable")[:k].tolist()
