"""Tree attention launches whose spare clusters prefetch the first chunks of
every split (D = 128, both kernels): back to back on one stream, with the
prefix lengths rewritten on the device between them, so that what is
prefetched was read from stale ones."""
import numpy as np
import pytest
import torch

from gpu_cases import AttnCase, assert_attention_close, ensure_built, i32
from paper_2512_21857_gb300 import binding as B

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    ensure_built()


@pytest.mark.parametrize("H,Hkv,sizes,max_kv,lens", [
    # 64-row kernel: four splits of 2.75 chunks (the last chunk is 8 rows), two heads a kv head, eight splits,
    # more room than eight clusters, four trees with one split each
    (32, 32, [64], 1160, [[1160], [0], [1], [127], [128], [129], [1153]]),
    (32, 16, [33], 1200, [[640], [1200]]),
    (16, 16, [7], 2433, [[2433], [64]]),
    (2, 2, [64], 1800, [[1800], [3]]),
    (32, 32, [64, 5, 33, 17], 700, [[700, 0, 129, 128], [1, 640, 0, 700]]),
    # 128-row kernel: two heads a CTA, trees of one and two tiles, two trees
    (32, 8, [64, 33], 3200, [[3200, 1], [127, 2049]]),
    (20, 20, [200], 1300, [[1300], [0]]),
    (20, 20, [256, 100], 1025, [[1025, 128], [0, 1025]]),
])
def test_prefetch_from_stale_lengths(H, Hkv, sizes, max_kv, lens):
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
