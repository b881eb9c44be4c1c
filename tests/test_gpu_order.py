"""Calls are ordered by their stream alone: inputs that the kernel just before a call writes -- a kernel of torch's, or the last
kernel of another call -- are read as written.  (The library's kernels are set up while their predecessors end; each has to
wait before its first read.)  No synchronisation inside a run; two sets of inputs take turns in the same buffers."""
import pytest
import torch

import _util as U
from paper_2606_23743_b200 import binding as B
from paper_2606_23743_b200.workloads import WORKLOADS, make_prologue_inputs, shrink

pytestmark = pytest.mark.gpu

W = {128: shrink(WORKLOADS["medium"], H=3, T=2, Hg=30, Wg=31, k=5),                    # N = 1860: 15 blocks, the last ragged
     64: shrink(WORKLOADS["medium"], H=3, T=2, Hg=30, Wg=31, k=9, block=64)}

# more than 64 blocks, the last ragged: scores and selection are kernels of their own
LONG = {128: shrink(WORKLOADS["medium"], H=3, T=9, Hg=30, Wg=31, k=9),                 # N = 8370: 66 blocks
        64: shrink(WORKLOADS["medium"], H=3, T=5, Hg=30, Wg=31, k=11, block=64)}       # N = 4650: 73 blocks


class Call:
    """A library call with the buffers it reads (`reads`, with two sets of contents) and writes (`writes`)."""

    def __init__(self, name, w):
        i32, u8 = torch.int32, torch.uint8

        def empty(*shape, dtype=torch.float32):
            return torch.empty(*shape, dtype=dtype, device="cuda")

        BH, made = w.B * w.H, [[x.cuda()[:, :, :w.N].contiguous() for x in U.host_inputs(w, seed=s)[0]] for s in (11, 12)]
        q, k, v = qkv = [torch.empty_like(x) for x in made[0]]
        o, lse, st = torch.empty_like(v), empty(w.B, w.H, w.N), torch.zeros(1, dtype=i32, device="cuda")
        p = B.make_problem(q, k, v, o, w.N, w.block)
        top, mass = B.make_select(0, w.k), B.make_select(1, w.k, 0.2)
        rp, ci, scores = empty(w.R + 1, dtype=i32), empty(w.R * w.k, dtype=i32), empty(w.B, w.H, w.Nb, w.Nb)
        sws = empty(max(256, B.select_workspace_bytes(p, top), B.select_workspace_bytes(p, mass)), dtype=u8)
        aws = empty(max(256, B.attn_workspace_bytes(p), B.attn_remainder_workspace_bytes(p, 1)), dtype=u8)
        q8, k8, qs, ks = e4m3 = [torch.empty_like(q, dtype=u8), torch.empty_like(k, dtype=u8), empty(w.B, w.H, w.Nb), empty(w.B, w.H, w.Nb)]
        p8 = B.make_problem(q8, k8, v, o, w.N, w.block, 0.0, True)
        f4 = [empty(BH, w.Nb * 128, 64, dtype=u8) for _ in range(2)] + [empty(BH, w.Nb, 1024, dtype=u8) for _ in range(2)] + \
             [empty(BH) for _ in range(2)]
        f4_ws = empty(max(256, 8 * BH), dtype=u8)
        qm, km = empty(w.B, w.H, w.Nb, w.d), empty(w.B, w.H, w.Nb, w.d)

        def route():
            B.block_select(p, top, q, k, rp, ci, sws, block_scores=scores)

        def e4m3_cast():
            B.quantize_qk_fp8(p, q, k, *e4m3)

        def sets(bufs, *makers):                       # contents that other calls make from the two sets of Q, K, V
            out = []
            for s in made:
                for b, x in zip(qkv, s):
                    b.copy_(x)
                for m in makers:
                    m()
                torch.cuda.synchronize()
                out.append([b.clone() for b in bufs])
            return out

        def remainder(order):
            B.block_sparse_attn_remainder_fwd(p, q, k, v, rp, ci, o, lse, st, order, aws, scores)

        self.reads, self.writes, self.sets = qkv, [o, lse], made
        if name == "block_select":
            self.writes, self.run = [rp, ci, scores], route
        elif name == "block_select_mass":
            self.writes, self.run = [rp], lambda: B.block_select(p, mass, q, k, rp, ci, sws)
        elif name == "block_select_noalloc":
            self.writes, self.run = [rp, ci], lambda: B.block_select_noalloc(p, top, q, k, rp, ci)
        elif name == "block_select_e4m3":
            self.reads, self.writes, self.sets = e4m3, [rp, ci], sets(e4m3, e4m3_cast)
            self.run = lambda: B.block_select(p8, top, q8, k8, rp, ci, sws, qs, ks)
        elif name == "pool_qk":
            self.writes, self.run = [qm, km], lambda: B.pool_qk(p, q, k, qm, km)
        elif name == "block_select_pooled":
            self.reads, self.writes, self.sets = [qm, km], [rp, ci], sets([qm, km], lambda: B.pool_qk(p, q, k, qm, km))
            self.run = lambda: B.block_select_pooled(p, top, qm, km, rp, ci, sws)
        elif name == "qk_norm_rope_pool":
            pro = [[x.cuda() for x in make_prologue_inputs(w, s)] for s in (1, 2)]
            pro[1][2:] = [x.flip(0).contiguous() for x in pro[1][2:]]                    # other rotary tables in the second set
            par = [torch.empty_like(x) for x in pro[0]]
            self.reads, self.sets = [q, k] + par, [s[:2] + t for s, t in zip(made, pro)]
            self.writes = [torch.empty_like(q), torch.empty_like(k), qm, km] + e4m3
            self.run = lambda: B.qk_norm_rope_pool(p, q, k, *par, 1e-6, *self.writes)
        elif name in ("attention", "attention_simt", "prepared"):
            self.reads = qkv + [rp, ci]
            self.sets = sets(self.reads, route)
            if name == "attention":
                self.run = lambda: B.block_sparse_attn_fwd(p, q, k, v, rp, ci, o, lse, st, workspace=aws)
            elif name == "attention_simt":
                self.run = lambda: B.block_sparse_attn_fwd_simt(p, q, k, v, rp, ci, o, lse, st)
            else:
                self.run = lambda: (B.attn_prepare_v(p, v, aws),
                                    B.block_sparse_attn_fwd_prepared(p, q, k, rp, ci, o, lse, st, workspace=aws))
        elif name == "dense":
            self.run = lambda: B.dense_attn_fwd(p, q, k, v, o, lse, st, workspace=aws)
        elif name == "attention_e4m3":
            self.reads = e4m3 + [v, rp, ci]
            self.sets = sets(self.reads, route, e4m3_cast)
            self.run = lambda: B.block_sparse_attn_fwd(p8, q8, k8, v, rp, ci, o, lse, st, qs, ks, workspace=aws)
        elif name == "attention_4bit":
            self.reads = f4 + [v, rp, ci]
            self.sets = sets(self.reads, route, lambda: B.quantize_qk_fp4(p, q, k, *f4, f4_ws))
            self.run = lambda: B.block_sparse_attn_fwd_fp4(p, *f4, v, rp, ci, o, lse, st, aws)
        elif name in ("remainder0", "remainder1"):
            self.reads = qkv + [rp, ci, scores]
            self.sets = sets(self.reads, route)
            self.run = lambda: remainder(int(name[-1]))
        elif name == "step_remainder":                 # whole steps: nothing but the library's kernels in between
            self.writes, self.run = [rp, ci, o, lse], lambda: (route(), remainder(1))
        elif name == "step":
            self.writes = [rp, ci, o, lse]
            self.run = lambda: (route(), B.block_sparse_attn_fwd(p, q, k, v, rp, ci, o, lse, st, workspace=aws))
        elif name == "step_e4m3":
            self.writes = e4m3 + [rp, ci, o, lse]
            self.run = lambda: (e4m3_cast(), B.block_select(p8, top, q8, k8, rp, ci, sws, qs, ks),
                                B.block_sparse_attn_fwd(p8, q8, k8, v, rp, ci, o, lse, st, qs, ks, workspace=aws))
        elif name == "step_4bit":
            self.writes = f4 + [rp, ci, o, lse]
            self.run = lambda: (route(), B.quantize_qk_fp4(p, q, k, *f4, f4_ws),
                                B.block_sparse_attn_fwd_fp4(p, *f4, v, rp, ci, o, lse, st, aws))
        elif name == "quantize_e4m3":
            self.writes, self.run = e4m3, e4m3_cast
        elif name == "quantize_e4m3_smooth":
            ws = empty(max(256, B.smooth_workspace_bytes(p)), dtype=u8)
            self.writes = e4m3 + [empty(w.B, w.H, w.d), empty(w.B, w.H, w.N)]
            self.run = lambda: B.quantize_qk_fp8_smooth_k(p, q, k, *self.writes, ws)
        elif name == "quantize_4bit":
            self.writes, self.run = f4, lambda: B.quantize_qk_fp4(p, q, k, *f4, f4_ws)
        else:
            m = 700
            picks = [torch.randperm(w.N, generator=torch.Generator().manual_seed(s))[:m].to(i32)[None].cuda() for s in (1, 2)]
            idx, part = torch.empty_like(picks[0]), empty(w.B, w.H, m, w.d, dtype=torch.bfloat16)
            self.reads = [q if name == "gather" else part, idx]
            self.sets = [[s[0] if name == "gather" else s[0][:, :, :m], i] for s, i in zip(made, picks)]
            self.writes = [part if name == "gather" else o]
            self.run = (lambda: B.gather_tokens(q, idx, part, st)) if name == "gather" else (lambda: B.scatter_tokens(part, idx, o, st))
        self.status = st

    def fill(self, i):
        for x in self.writes:
            x.view(torch.uint8).fill_(0x55)
        for b, x in zip(self.reads, self.sets[i]):
            b.copy_(x)


NAMES = ["block_select", "block_select_mass", "block_select_noalloc", "block_select_e4m3", "pool_qk", "block_select_pooled",
         "qk_norm_rope_pool", "attention", "attention_simt", "prepared", "dense", "attention_e4m3", "remainder0", "remainder1", "step",
         "step_remainder", "step_e4m3", "quantize_e4m3", "quantize_e4m3_smooth", "gather", "scatter"]
CASES = [(n, b) for n in NAMES for b in (128, 64)] + [(n, 128) for n in ("quantize_4bit", "attention_4bit", "step_4bit")]


@pytest.mark.parametrize("name,block", CASES)
def test_inputs_written_just_before_a_call(name, block):
    _check(Call(name, W[block]))


@pytest.mark.parametrize("name,block", [(n, b) for n in ("block_select", "block_select_mass", "block_select_noalloc", "block_select_e4m3",
                                                         "block_select_pooled", "step", "step_remainder", "step_e4m3") for b in (128, 64)] +
                         [("step_4bit", 128)])
def test_inputs_written_just_before_a_call_of_many_blocks(name, block):
    _check(Call(name, LONG[block]))


def _check(c):
    want = []
    for i in range(2):
        c.fill(i)
        torch.cuda.synchronize()
        c.run()
        torch.cuda.synchronize()
        want.append([x.clone() for x in c.writes])
    assert any(not torch.equal(a.view(torch.uint8), b.view(torch.uint8)) for a, b in zip(*want))     # the sets do differ
    busy = torch.empty(1 << 28, dtype=torch.uint8, device="cuda")
    got = []
    torch.cuda.synchronize()
    for i in range(6):
        for _ in range(3):
            busy.fill_(i)                              # the host gets ahead of the GPU, so that what follows runs back to back
        c.fill(i & 1)
        c.run()
        got.append([x.clone() for x in c.writes])
    torch.cuda.synchronize()
    assert int(c.status.item()) == 0
    for i, outs in enumerate(got):
        for a, b in zip(outs, want[i & 1]):
            assert torch.equal(a.view(torch.uint8), b.view(torch.uint8)), i
