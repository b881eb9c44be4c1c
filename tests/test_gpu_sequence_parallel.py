"""The sequence-parallel wrapper on one GPU: a one-rank NCCL group, so that the CUDA `attend` callable and
the NCCL exchange calls run for real (the multi-rank exchange itself is covered on CPU with gloo)."""
import socket

import pytest
import torch
import torch.distributed as dist

import _util as U
from paper_2606_23743_b200 import binding as B
from paper_2606_23743_b200 import sequence_parallel as SP
from paper_2606_23743_b200.workloads import WORKLOADS, bf16_bits, shrink

pytestmark = pytest.mark.gpu


def test_one_rank_group_matches_the_direct_path_and_the_oracle():
    s = socket.socket(); s.bind(("127.0.0.1", 0)); port = s.getsockname()[1]; s.close()
    dist.init_process_group("nccl", init_method=f"tcp://127.0.0.1:{port}", rank=0, world_size=1)
    try:
        w = shrink(WORKLOADS["large"], H=2, T=2)
        (q, k, v), (qb, kb, vb) = U.host_inputs(w)
        qd, kd, vd = (U.dev(x)[:, :, :w.N].contiguous() for x in (q, k, v))
        sel = B.make_select(w.mode, w.k, w.tau)
        attend = SP.sparse_attend(sel, w.block)
        o = SP.sequence_parallel_attention(qd, kd, vd, SP.even_shards(w.N, 1), attend)
        torch.cuda.synchronize()
        assert int(attend.status.item()) == 0                 # what the kernels reported is not dropped
        rp, ci, _ = U.gpu_select(w, U.dev(q), U.dev(k))
        o_direct, _, st = U.gpu_attn(w, U.dev(q), U.dev(k), U.dev(v), rp, ci)
        assert st == 0 and torch.equal(o, o_direct[:, :, :w.N])
        U.check_attn_vs_oracle(w, qb, kb, vb, rp, ci, o, None, U.sample_rows(w.R, w.Nb, 6))
    finally:
        dist.destroy_process_group()


def test_attend_does_not_depend_on_what_its_buffers_held(monkeypatch):
    """A NaN token leaves its query block without scores, and its key block without candidates that k = Nb counts on: the output
    is that of index arrays that were cleared, whatever the allocator hands out."""
    w = shrink(WORKLOADS["medium"], H=2, T=1, k=8)                 # 8 blocks, all of them asked for
    (q, k, v), _ = U.host_inputs(w)
    qd, kd, vd = (U.dev(x)[:, :, :w.N].contiguous() for x in (q, k, v))
    qd[0, 0, 300, 5] = float("nan")
    kd[0, 1, 700, 9] = float("nan")
    sel = B.make_select(0, w.k)
    p = B.make_problem(qd, kd, vd, torch.empty_like(vd), w.N, w.block)
    rp, ci = (torch.zeros(n, dtype=torch.int32, device="cuda") for n in (w.R + 1, B.select_max_nnz(p, sel)))
    B.block_select(p, sel, qd, kd, rp, ci, torch.empty(B.select_workspace_bytes(p, sel), dtype=torch.uint8, device="cuda"))
    want, _, st = U.gpu_attn(w, qd, kd, vd, rp, ci)
    assert st == 0
    attend = SP.sparse_attend(sel, w.block)
    empty = torch.empty
    for junk in (3, 7):                                            # (valid indices: a stale list would go unnoticed)
        def held(*size, dtype=None, **kw):                         # memory that an earlier call has used
            x = empty(*size, dtype=dtype, **kw)
            return x.fill_(junk) if dtype == torch.int32 else x
        monkeypatch.setattr(torch, "empty", held)
        o = attend(qd, kd, vd)
        monkeypatch.setattr(torch, "empty", empty)
        assert int(attend.status.item()) == 0
        assert torch.equal(o.view(torch.int16), want[:, :, :w.N].view(torch.int16))
