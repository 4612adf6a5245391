"""Failure detection without a GPU fault: a bounded device-side wait runs
out and is reported through the device error word, the call returns
cleanly, and the device stays usable (the next call matches the oracle)."""
import pytest

import oracle
from gpu_cases import AttnCase, assert_attention_close, ensure_built, run_accept_gpu
from paper_2512_21857_gb300 import binding as B
from paper_2512_21857_gb300 import synth
from test_parity_accept_compact import ACCEPT_MARGIN, SAMPLE_MARGIN, compare, make_rows

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    ensure_built()


def test_attention_wait_that_runs_out_is_reported_and_the_device_stays_usable():
    # 16 heads x 8 key splits (clusters of 8 CTAs, 2-3 chunks each): with a
    # bound of one poll, waits for loads and products that take microseconds
    # give up.
    case = AttnCase([64], [2400], 16, 16, 128, seed=55)
    ref, _ = case.run_oracle()
    B.adt_get_device_error()
    try:
        B.adt_testing_set_wait_limit(1)
        case.run_gpu()  # the launch itself succeeds; its outputs are unspecified
    finally:
        B.adt_testing_set_wait_limit(0)
    bits = B.adt_get_device_error()
    assert bits & B.DEVERR_TIMEOUT
    assert B.adt_get_device_error() == 0  # read and cleared
    for _ in range(2):
        got, _, _ = case.run_gpu()
        assert B.adt_get_device_error() == 0
        assert_attention_close(got, ref)


@pytest.mark.parametrize("V", [16384, 65536])  # 8 and 16 CTAs a tree
@pytest.mark.parametrize("mode", [B.ACCEPT_SPEC, B.ACCEPT_SPEC_DET])
def test_acceptance_wait_that_runs_out_is_reported_and_the_device_stays_usable(mode, V):
    for seed in range(70, 90):
        tb = synth.tree_batch([64, 33, 50], V, seed, max_depth=6, max_children=12)
        target, draft = make_rows(tb, V, seed, 0.3)
        ua, us = (synth.uniforms(len(tb.tokens), seed, name) for name in ("ua", "us"))
        args = (target, draft if mode == B.ACCEPT_SPEC else None, tb, mode, ua, us)
        res = oracle.tree_accept(target, draft, tb.tokens, tb.parents, tb.node_offsets, mode, ua, us)
        if res["accept_margin"] > ACCEPT_MARGIN and res["sample_margin"] > SAMPLE_MARGIN:
            break
    B.adt_get_device_error()
    for _ in range(20):
        try:
            B.adt_testing_set_wait_limit(1)
            path, alen, _ = run_accept_gpu(*args)
        finally:
            B.adt_testing_set_wait_limit(0)
        assert B.adt_get_device_error() == B.DEVERR_TIMEOUT
        assert (path[:, 0] == 0).all() and (path[:, 1:] == -1).all() and (alen == 0).all()
        compare(tb, res, *run_accept_gpu(*args))
        assert B.adt_get_device_error() == 0
