"""Tree attention launches whose spare clusters prefetch the first chunks of
every split (D = 128, both kernels), which they do from prefix lengths that an
earlier launch may still be writing."""
import numpy as np
import pytest
import torch

from gpu_cases import AttnCase, assert_attention_close, ensure_built, i32
from paper_2512_21857_gb300 import binding as B

pytestmark = pytest.mark.gpu

SHAPES = [
    # H, Hkv, tree sizes, max_kv, prefix lengths of the calls, (rows, thread blocks that share the keys)
    # 64-row kernel: four splits of 2.75 chunks (the last chunk is 8 rows), two heads a kv head, six splits, eight
    # splits, four trees with one split each
    (32, 32, [64], 1160, [[1160], [0], [1], [127], [128], [129], [1153]], (64, 4)),
    (32, 16, [33], 1200, [[640], [1200]], (64, 4)),
    (16, 16, [7], 2433, [[2433], [64]], (64, 6)),
    (10, 10, [64], 2500, [[2500], [3]], (64, 8)),
    (32, 32, [64, 5, 33, 17], 700, [[700, 0, 129, 128], [1, 640, 0, 700]], (64, 1)),
    # 128-row kernel, which prefetches from four chunks a split on: two heads a CTA, trees of one and two tiles, two trees
    (32, 8, [64, 33], 3200, [[3200, 1], [127, 2049]], (128, 4)),
    (20, 20, [200], 1700, [[1700], [0]], (128, 6)),
    (20, 20, [256, 100], 1025, [[1025, 128], [0, 1025]], (128, 2)),
]


@pytest.fixture(scope="module", autouse=True)
def _built():
    ensure_built()


def _prefetches(H, Hkv, sizes, max_kv, lens, rows, blocks):
    """The launch is the one the case is there for, and some call prefetches."""
    plan = B.adt_testing_attn_plan(len(sizes), H, Hkv, 128, max(sizes), max_kv)
    assert plan[:2] == (rows, blocks) and plan[2] > 0, plan
    if rows == 128:
        splits = [blocks // (1 if H > Hkv else -(-n // 128)) for n in sizes]
        assert any(L >= 4 * 128 * s for length in lens for L, s in zip(length, splits))


@pytest.mark.parametrize("H,Hkv,sizes,max_kv,lens,plan", SHAPES)
def test_launches_back_to_back(H, Hkv, sizes, max_kv, lens, plan):
    """Calls on one stream, the prefix lengths rewritten between them by a copy."""
    _prefetches(H, Hkv, sizes, max_kv, lens, *plan)
    nb, n = len(sizes), max(sizes)
    cases = [AttnCase(sizes, L, H, Hkv, 128, seed=7 * sum(L) + H, lmax=max_kv, max_depth=8, max_children=39)
             for L in lens]
    c0 = cases[0]
    dev = "cuda"
    ws = B.zeroed_workspace(B.adt_tree_attn_workspace_size(nb, H, 128, n, max_kv))
    kv_len = i32([max_kv] * nb)
    ins = [(c.q.to(dev), c.kc.to(dev), c.vc.to(dev), c.kt.to(dev), c.vt.to(dev), i32(c.tb.parents),
            i32(c.tb.node_offsets), i32(c.kv_lens)) for c in cases]
    outs = [torch.empty((c.ntot, H, 128), dtype=torch.bfloat16, device=dev) for c in cases]
    torch.cuda.synchronize()
    for (q, kc, vc, kt, vt, par, offs, length), out in zip(ins, outs):
        kv_len.copy_(length)
        for _ in range(3):  # the second and third overlap the one before
            B.adt_tree_attn(q, kc, vc, kv_len, kt, vt, par, offs, B=nb, H=H, Hkv=Hkv, D=128, max_nodes=n, max_kv=max_kv,
                            softmax_scale=c0.scale, out=out, workspace=ws)
    torch.cuda.synchronize()
    assert B.adt_get_device_error() == 0
    for c, out in zip(cases, outs):
        assert_attention_close(out.float().cpu().numpy().astype(np.float64), c.run_oracle()[0])


@pytest.mark.parametrize("stale", [0, 1, 2 ** 30, -5])
@pytest.mark.parametrize("H,Hkv,sizes,max_kv,lens,plan", [SHAPES[0], SHAPES[4], SHAPES[5], SHAPES[6]])
def test_prefetch_from_stale_lengths(H, Hkv, sizes, max_kv, lens, plan, stale):
    """Commit, then attention over the lengths it writes: adt_kv_compact lets its
    dependents start before it writes them (and the cache rows they cover), so
    the prefetching clusters may read what the array held before."""
    nb, n, D = len(sizes), max(sizes), 128
    commit = 6
    prefix = [max(0, L - commit) for L in lens[0]]
    after = [L + commit for L in prefix]
    max_kv += commit
    _prefetches(H, Hkv, sizes, max_kv, [after], *plan)
    c = AttnCase(sizes, after, H, Hkv, D, seed=17 * sum(after) + H, lmax=max_kv, max_depth=8, max_children=39)
    g = torch.Generator().manual_seed(3)
    old_k, old_v = (torch.randn((nb * commit, Hkv, D), generator=g).to(torch.bfloat16) for _ in range(2))
    path = i32(np.tile(np.arange(commit), (nb, 1)))
    dev = "cuda"
    kc0, vc0 = c.kc.to(dev), c.vc.to(dev)
    for b, L in enumerate(prefix):
        c.kc[b, :, L:L + commit] = old_k[b * commit:(b + 1) * commit].transpose(0, 1)
        c.vc[b, :, L:L + commit] = old_v[b * commit:(b + 1) * commit].transpose(0, 1)
    kc, vc, kv, kv_out = torch.empty_like(kc0), torch.empty_like(vc0), i32(prefix), i32([0] * nb)
    q, kt, vt, par, offs = c.q.to(dev), c.kt.to(dev), c.vt.to(dev), i32(c.tb.parents), i32(c.tb.node_offsets)
    old_k, old_v, old_offs, alen = old_k.to(dev), old_v.to(dev), i32(np.arange(nb + 1) * commit), i32([commit - 1] * nb)
    out = torch.empty((8, c.ntot, H, D), dtype=torch.bfloat16, device=dev)
    ws = B.zeroed_workspace(B.adt_tree_attn_workspace_size(nb, H, D, n, max_kv))
    for i in range(len(out)):
        kc.copy_(kc0)
        vc.copy_(vc0)
        kv_out.fill_(stale)
        B.adt_kv_compact(kc, vc, kv, kv_out, old_k, old_v, old_offs, path, commit, alen, B=nb, Hkv=Hkv, D=D,
                         num_layers=1, max_kv=max_kv, cache_layer_stride=0, cache_stride_b=kc.stride(0),
                         cache_stride_h=kc.stride(1), tree_layer_stride=0)
        B.adt_tree_attn(q, kc, vc, kv_out, kt, vt, par, offs, B=nb, H=H, Hkv=Hkv, D=D, max_nodes=n,
                        max_kv=max_kv, softmax_scale=c.scale, out=out[i], workspace=ws)
    torch.cuda.synchronize()
    assert B.adt_get_device_error() == 0
    assert kv_out.tolist() == after
    assert_attention_close(out[0].float().cpu().numpy().astype(np.float64), c.run_oracle()[0])
    assert torch.equal(out, out[:1].expand_as(out))


@pytest.mark.parametrize("H,Hkv,sizes,max_kv,plan", [
    (32, 32, [64], 1160, (64, 4)), (32, 8, [64, 33], 3200, (128, 4)), (20, 20, [200], 1700, (128, 6)),
])
def test_caches_with_gaps(H, Hkv, sizes, max_kv, plan):
    """Cache strides larger than the packed ones, NaN in what lies between."""
    lens = [max_kv] + [max_kv // 3] * (len(sizes) - 1)
    _prefetches(H, Hkv, sizes, max_kv, [lens], *plan)
    c = AttnCase(sizes, lens, H, Hkv, 128, seed=max_kv, lmax=max_kv, max_depth=8, max_children=39)
    nb, n = len(sizes), max(sizes)
    big = [torch.full((nb, Hkv + 1, max_kv + 24, 128), float("nan"), dtype=torch.bfloat16, device="cuda") for _ in "kv"]
    kc, vc = (t[:, :Hkv, :max_kv] for t in big)
    kc.copy_(c.kc)
    vc.copy_(c.vc)
    out = torch.empty((3, c.ntot, H, 128), dtype=torch.bfloat16, device="cuda")
    args = [t.cuda() for t in (c.kt, c.vt)] + [i32(c.tb.parents), i32(c.tb.node_offsets)]
    q, kv = c.q.cuda(), i32(lens)
    ws = B.zeroed_workspace(B.adt_tree_attn_workspace_size(nb, H, 128, n, max_kv))
    for o in out:
        B.adt_tree_attn(q, kc, vc, kv, *args, B=nb, H=H, Hkv=Hkv, D=128, max_nodes=n, max_kv=max_kv,
                        softmax_scale=c.scale, out=o, workspace=ws)
    torch.cuda.synchronize()
    ref = c.run_oracle()[0]
    for o in out:
        assert_attention_close(o.float().cpu().numpy().astype(np.float64), ref)
