"""Tree attention over 128-row tiles: the launches that take it (long key
ranges per CTA; two heads of a kv head per CTA, or trees of more than 64
nodes), at the edges of its tiles, chunks of 128 keys, 32-key quarters and
16-key product steps, with one split and with several."""
import numpy as np
import pytest
import torch

from gpu_cases import LSE_ATOL, AttnCase, assert_attention_close, ensure_built, i32
from paper_2512_21857_gb300 import binding as B

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    ensure_built()


def _check(case, max_nodes):
    got, lse, _ = case.run_gpu(max_nodes=max_nodes)
    ref, ref_lse = case.run_oracle()
    assert_attention_close(got, ref)
    assert np.abs(lse - ref_lse).max() < LSE_ATOL


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("sizes,kv,H,Hkv,max_nodes", [
    # two heads a CTA: one split (80 groups), four splits (32 groups)
    ([1, 64, 33, 7, 26] * 4, [0, 1, 640, 129, 127] * 4, 8, 4, 64),
    ([64, 33, 5, 17], [1537, 1403, 128, 0], 16, 8, 64),
    # trees of up to 256 nodes: dealt to one or two tiles of six CTAs; tiles of their own (80 groups)
    ([200], [700], 20, 20, 256),
    ([41], [1203], 20, 20, 256),
    ([129], [895], 20, 20, 200),
    ([256, 41, 128, 1], [320, 0, 97, 33], 20, 20, 256),
    ([100, 65], [650, 17], 32, 8, 100),
])
def test_wide_tiles_match_oracle(sizes, kv, H, Hkv, max_nodes, D):
    _check(AttnCase(sizes, kv, H, Hkv, D, seed=sum(sizes) + D, max_depth=10, max_children=39, lmax=max(max(kv), 700)),
           max_nodes)


def test_wide_more_trees_than_the_launch_orders():
    """33 trees: past 32 the launch takes them as they come."""
    sizes = [1 + (7 * i) % 64 for i in range(33)]
    kv = [(97 * i) % 700 for i in range(33)]
    assert B.adt_testing_attn_plan(33, 8, 4, 128, 64, 900)[0] == 128
    case = AttnCase(sizes, kv, 8, 4, 128, seed=33, max_depth=10, max_children=8, lmax=900)
    got, _, _ = case.run_gpu(max_nodes=64, max_kv=900)
    assert_attention_close(got, case.run_oracle()[0])


@pytest.mark.parametrize("kv", [769, 783, 784, 785, 800, 801, 864, 895])
def test_wide_prefix_ends(kv):
    """Every kind of end of the last chunk; whatever the cache holds past it (NaN) has no effect."""
    case = AttnCase([70, 128], [kv, kv - 640], 20, 20, 64, seed=kv, lmax=960, max_depth=10, max_children=39)
    ref, _ = case.run_oracle()
    for b, L in enumerate(case.kv_lens):
        case.kc[b, :, L:] = float("nan")
        case.vc[b, :, L:] = float("nan")
    got, _, _ = case.run_gpu(max_nodes=128, max_kv=960)
    assert_attention_close(got, ref)


def test_wide_tiles_with_few_rows_repeat():
    """Tiles whose last warps have no rows, one split each, prefixes that end
    within a 16-key step: those warps run ahead of the others to the end of
    the prefix, where they help to clear V rows in a ring of two slots."""
    case = AttnCase([48, 33, 61, 86] * 2, [900, 1140, 517, 777] * 2, 20, 20, 128, seed=21, max_depth=10,
                    max_children=39)
    ref, _ = case.run_oracle()
    for _ in range(30):
        got, _, _ = case.run_gpu(max_nodes=128)
        assert_attention_close(got, ref)


def test_wide_chain_of_256_nodes():
    _check(AttnCase([256], [640], 20, 20, 128, seed=3, chain=True), 256)


@pytest.mark.parametrize("D", [64, 128])
def test_wide_scores_that_grow(D):
    """Keys whose scores rise by far more than 2^8 from chunk to chunk: the
    running maximum passes from one softmax group to the other and O is scaled."""
    case = AttnCase([200, 130, 256, 77], [1000, 900, 640, 3], 20, 20, D, seed=9, max_depth=10, max_children=39)
    ramp = torch.linspace(0.0, 60.0, case.lmax)[None, None, :, None]
    unit = torch.nn.functional.normalize(case.q[:, :, :].float().mean(0), dim=-1)
    case.kc = (case.kc.float() + ramp * unit[None, :, None, :]).to(torch.bfloat16)
    case.q = (case.q.float() + 4.0 * unit[None]).to(torch.bfloat16)
    _check(case, 256)


def test_wide_bad_tree_sets_device_error():
    case = AttnCase([150], [700], 20, 20, 64, seed=5, max_depth=10, max_children=39)
    case.tb.parents[140] = 145
    B.adt_get_device_error()
    case.run_gpu(max_nodes=256)
    assert B.adt_get_device_error() & B.DEVERR_BAD_TREE
    case.tb.parents[140] = 0
    _check(case, 256)
    assert B.adt_get_device_error() == 0


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("sizes,kv,H,Hkv,max_nodes", [
    ([150, 70], [700, 300], 20, 20, 256),                  # key splits of two tiles
    ([64, 33, 5, 17], [1537, 1403, 128, 0], 16, 8, 64),    # two heads a CTA, four splits
    ([256, 41, 128, 1], [320, 0, 97, 33], 20, 20, 256),    # one split a tile
])
def test_wide_bad_tree_is_skipped(sizes, kv, H, Hkv, max_nodes, D):
    """A malformed tree's rows stay as they were, in every tile and split; the
    other trees of the call are computed."""
    case = AttnCase(sizes, kv, H, Hkv, D, seed=sum(sizes) + D, max_depth=10, max_children=39, lmax=max(max(kv), 700))
    ref, ref_lse = case.run_oracle()
    n0 = sizes[0]
    for at, parent in ((n0 - 1, n0 - 1), (1, -1), (0, 0)):
        good = int(case.tb.parents[at])
        case.tb.parents[at] = parent
        out = torch.full((case.ntot, H, D), 7.0, dtype=torch.bfloat16, device="cuda")
        lse = torch.full((case.ntot, H), 7.0, dtype=torch.float32, device="cuda")
        B.adt_get_device_error()
        B.adt_tree_attn(case.q.cuda(), case.kc.cuda(), case.vc.cuda(), i32(kv), case.kt.cuda(), case.vt.cuda(),
                        i32(case.tb.parents), i32(case.tb.node_offsets), B=case.B, H=H, Hkv=Hkv, D=D,
                        max_nodes=max_nodes, max_kv=max(kv), softmax_scale=case.scale, out=out, lse=lse,
                        workspace=B.zeroed_workspace(B.adt_tree_attn_workspace_size(case.B, H, D, max_nodes, max(kv))))
        assert B.adt_get_device_error() == B.DEVERR_BAD_TREE
        assert (out[:n0] == 7.0).all() and (lse[:n0] == 7.0).all()
        assert_attention_close(out[n0:].float().cpu().numpy().astype(np.float64), ref[n0:])
        assert np.abs(lse[n0:].cpu().numpy() - ref_lse[n0:]).max() < LSE_ATOL
        case.tb.parents[at] = good


def test_wide_wait_that_runs_out_is_reported():
    case = AttnCase([150], [700], 20, 20, 128, seed=6, max_depth=10, max_children=39)
    B.adt_get_device_error()
    B.adt_testing_set_wait_limit(1)
    try:
        case.run_gpu(max_nodes=256)
        assert B.adt_get_device_error() & B.DEVERR_TIMEOUT
    finally:
        B.adt_testing_set_wait_limit(0)
    _check(case, 256)
    assert B.adt_get_device_error() == 0
