"""First calls of the acceptance walk from several host threads at once, each
with another vocabulary: a kernel's launch limits do not depend on the order of
the calls."""
import os
import subprocess
import sys

import pytest

from gpu_cases import ensure_built

pytestmark = pytest.mark.gpu

SCRIPT = """
import threading
import numpy as np
import torch
import oracle
from gpu_cases import f32, f32_rows, i32
from paper_2512_21857_gb300 import binding as B
from paper_2512_21857_gb300 import synth
from test_parity_accept_compact import compare, make_rows

jobs = []
for i, V in enumerate([4096, 60000, 8192, 49152, 16384, 65536, 12288, 32768] * 2):
    mode = B.ACCEPT_SPEC if i < 8 else B.ACCEPT_SPEC_DET
    tb = synth.tree_batch([12, 9], V, i, max_depth=4, max_children=4)
    target, draft = make_rows(tb, V, i, 0.3)
    ua, us = (synth.uniforms(len(tb.tokens), i, n) for n in ("ua", "us"))
    jobs.append((tb, oracle.tree_accept(target, draft, tb.tokens, tb.parents, tb.node_offsets, mode, ua, us),
                 (f32_rows(target), f32_rows(draft) if mode == B.ACCEPT_SPEC else None, i32(tb.tokens),
                  i32(tb.parents), i32(tb.node_offsets)),
                 dict(B=2, V=V, max_nodes=12, mode=mode, u_accept=f32(ua), u_sample=f32(us), max_path=8,
                      path=torch.empty((2, 8), dtype=torch.int32, device="cuda"),
                      accept_len=torch.empty(2, dtype=torch.int32, device="cuda"),
                      bonus_token=torch.empty(2, dtype=torch.int32, device="cuda"),
                      stream=torch.cuda.Stream())))
B.lib()
torch.cuda.synchronize()
start, failed = threading.Barrier(len(jobs)), []

def call(args, kw):
    start.wait()
    try:
        B.adt_tree_accept(*args, **kw)
    except B.AdtError as e:
        failed.append((kw["V"], str(e)))

threads = [threading.Thread(target=call, args=job[2:]) for job in jobs]
for t in threads:
    t.start()
for t in threads:
    t.join()
torch.cuda.synchronize()
assert not failed, failed
for tb, res, _, kw in jobs:
    if res["min_margin"] > 1e-9:
        compare(tb, res, kw["path"].cpu().numpy(), kw["accept_len"].cpu().numpy(), kw["bonus_token"].cpu().numpy())
"""


def test_first_calls_from_several_threads():
    ensure_built()
    tests = os.path.dirname(os.path.abspath(__file__))
    env = dict(os.environ, PYTHONPATH=os.pathsep.join([os.path.dirname(tests), tests]))
    for _ in range(3):
        r = subprocess.run([sys.executable, "-c", SCRIPT], env=env, capture_output=True, text=True, timeout=300)
        assert r.returncode == 0, r.stderr[-2000:]
