"""The give-up paths: in each form of the attention kernel a row's K tiles after the first are withheld (test switch), in the kernels of the
remainder's first-order term some of their loads; the bounded waits run out, and every role leaves.  Nothing faults or hangs."""
import time

import pytest
import torch

import _util as U
from paper_2606_23743_b200 import binding as B
from paper_2606_23743_b200.workloads import WORKLOADS, shrink
from test_gpu_fp4 import gpu_attn_fp4, gpu_quantize4
from test_gpu_fp8 import _quantize
from test_gpu_remainder import gpu_remainder

pytestmark = pytest.mark.gpu


def _call(form, block):
    """A call of the form with rows of several tiles, as a function that makes it again: -> (o, lse, status)."""
    w = shrink(WORKLOADS["medium"], H=1, T=2, block=block, k=6)               # 2 048 tokens: a row per CTA
    (q, k, v), _ = U.host_inputs(w)
    q, k, v = U.dev(q), U.dev(k), U.dev(v)
    rp, ci, scores = U.gpu_select(w, q, k, want_scores=True)
    if form == "bf16":
        return lambda: U.gpu_attn(w, q, k, v, rp, ci)
    if form == "dense":
        return lambda: U.gpu_attn(w, q, k, v, None, None, dense=True)
    if form == "e4m3":
        q8, k8, qs, ks = _quantize(w, q, k)
        return lambda: U.gpu_attn(w, q8, k8, v, rp, ci, q_scale=qs, k_scale=ks, fp8=True)
    if form == "4-bit":
        codes = gpu_quantize4(w, q, k)
        return lambda: gpu_attn_fp4(w, codes, v, rp, ci)
    return lambda: gpu_remainder(w, q, k, v, rp, ci, 1, scores=scores)


@pytest.mark.parametrize("form,block", [("bf16", 128), ("bf16", 64), ("dense", 128), ("e4m3", 128), ("e4m3", 64), ("4-bit", 128),
                                        ("remainder", 128), ("remainder", 64)])
def test_a_starved_row_is_reported_and_not_stored(form, block):
    """No tile after a row's first exists: no MMA may be issued for it, no barrier told that it was, and so no row stored."""
    call = _call(form, block)
    want, want_lse, st = call()
    assert st == 0
    try:
        B.debug_set_wait_limit(100_000_000)                                   # about 50 ms
        B.debug_set_mode(16)
        o, lse, st = call()
    finally:
        B.debug_set_mode(0)
        B.debug_set_wait_limit(0)
    assert st == B.SVA_DEV_TIMEOUT
    assert (o == 7.0).all() and (lse == 7.0).all()                            # (as the caller left them)
    o, lse, st = call()                                                       # the context and the next call are intact
    assert st == 0 and torch.equal(o, want) and torch.equal(lse, want_lse)


@pytest.mark.parametrize("block", [128, 64])
@pytest.mark.parametrize("switch", [256, 512], ids=["covariances", "aggregation"])
def test_starved_first_order_kernels_give_up(switch, block):
    """A CTA of either kernel whose load never arrives reports it and leaves, with stores of its first tiles under way, in the time that the
    limit allows (the default limit is thirty times that)."""
    w = shrink(WORKLOADS["medium"], H=4, T=2, block=block, k=6)               # (four heads: several column tiles per CTA)
    (q, k, v), _ = U.host_inputs(w)
    q, k, v = U.dev(q), U.dev(k), U.dev(v)
    rp, ci, scores = U.gpu_select(w, q, k, want_scores=True)
    want, want_lse, st = gpu_remainder(w, q, k, v, rp, ci, 1, scores=scores)
    assert st == 0
    try:
        B.debug_set_wait_limit(100_000_000)                                   # about 50 ms
        B.debug_set_mode(switch)
        t0 = time.monotonic()
        _, _, st = gpu_remainder(w, q, k, v, rp, ci, 1, scores=scores)
        took = time.monotonic() - t0
    finally:
        B.debug_set_mode(0)
        B.debug_set_wait_limit(0)
    assert st == B.SVA_DEV_TIMEOUT and 0.04 < took < 1.0, took
    o, lse, st = gpu_remainder(w, q, k, v, rp, ci, 1, scores=scores)
    assert st == 0 and torch.equal(o, want) and torch.equal(lse, want_lse)
