"""The work that users of this library have it do, as measurable cases.

A case is one self-attention call of a video diffusion transformer on one GPU, through the entry points of
`paper_2606_23743_b200.binding`: routing, then attention over the routed blocks (or dense attention), with the options
a deployment switches on -- e4m3 or 4-bit Q/K, K smoothing, the fused QK-norm + RoPE prologue, the approximate
remainder of the dropped blocks, a pruned token subset.  Buffers, workspaces and the problem description are kept by
the caller, as a denoising loop keeps them; only `attend` cases go through the convenience callable
`sequence_parallel.sparse_attend`, which allocates per call.

Keys of a case:
  B, H, d            batch items, heads, head dimension
  T, Hg, Wg          video latent grid; N = T * Hg * Wg tokens, w fastest
  block, mode, k, tau, window   routing rule: top-k (mode 0) or cumulative mass >= tau capped at k (mode 1); a forced
                     3 x 3 neighbour window on the (frame, strip) block grid
  qk                 "bf16", "fp8" (e4m3 codes made in the pass), "fp4" (block-scaled e2m1 codes made in the pass)
  form               "sparse", "dense", or "attend" (the convenience callable)
  remainder          -1 none, else the order (0, 1) of the approximate remainder
  prologue, smooth   fused QK-norm + RoPE prologue in front; mean key taken out of K before the e4m3 cast
  keep               share of the tokens that attention sees (token pruning); 1.0 = all of them
  layout             "heads" [B, H, N, d]; "tokens" [B, N, H, d]; "packed": Q, K, V as views of one [B, N, 3, H, d]
  qk_mult            Q and K multiplied by this (sharper scores)
"""
import math

import torch

from paper_2606_23743_b200 import binding as sva
from paper_2606_23743_b200.sequence_parallel import sparse_attend
from paper_2606_23743_b200.workloads import WORKLOADS, Workload, make_prologue_inputs

BASE = dict(B=1, H=16, d=128, T=8, Hg=32, Wg=32, block=128, mode=0, k=16, tau=1.0, window=False, qk="bf16", form="sparse",
            remainder=-1, prologue=False, smooth=False, keep=1.0, layout="heads", qk_mult=1.0)
GRID = ("B", "H", "d", "T", "Hg", "Wg", "block", "mode", "k", "tau", "qk_mult")


def _from_workload(name, workload, **options):
    w = WORKLOADS[workload]
    return dict(BASE, name=name, window=w.win_t >= 0, **{g: getattr(w, g) for g in GRID}, **options)


def listed():
    return [
        # the smallest call: a preview-sized clip, two heads; launches and host calls are what it consists of
        _from_workload("tiny_d64_b64", "tiny"),
        # a short clip through the callable that allocates for its caller; ragged length, mass rule, packed QKV projection
        dict(BASE, name="small_attend_ragged", H=12, T=6, Hg=30, Wg=31, mode=1, k=12, tau=0.9, form="attend", layout="packed"),
        # an ordinary low-resolution clip
        _from_workload("medium", "medium"),
        # the layers a deployment keeps dense, at the same size
        _from_workload("medium_dense", "medium", form="dense"),
        # the headline size: 32 760 tokens, 15 % of the key blocks by cumulative mass
        _from_workload("large", "large"),
        # a classifier-free-guidance pair of a large model: top-k with the forced neighbour window; the largest call
        _from_workload("xl", "xl"),
        # the 8-bit variant of the headline size
        _from_workload("large_fp8", "large_fp8", qk="fp8"),
        # the 4-bit variant behind the fused prologue, which also writes the block means that routing takes
        _from_workload("large_prologue_fp4", "large", qk="fp4", prologue=True),
        # the paper's deployment preset: 64-token blocks, about 10 % of them kept ...
        _from_workload("large_b64", "large_b64"),
        # ... and with its approximate remainder switched on
        _from_workload("large_b64_remainder0", "large_b64", remainder=0),
        # the remainder with its first-order term, 128-token blocks, tensors as the projection leaves them
        dict(BASE, name="mid_remainder1_tokens", H=20, T=13, Hg=30, Wg=45, mode=1, k=22, tau=0.9, remainder=1, layout="tokens"),
        # token pruning: half of the tokens are gathered, routed, attended with 64-token blocks and scattered back
        dict(_from_workload("large_pruned_b64", "large_b64"), keep=0.5, k=26, layout="tokens"),
    ]


def _workload(case):
    return Workload("case", 0, case["B"], case["H"], case["d"], case["T"], case["Hg"], case["Wg"], case["block"], case["mode"],
                    case["k"], tau=case["tau"], win_t=1 if case["window"] else -1, win_s=1 if case["window"] else -1,
                    qk_mult=case["qk_mult"])


def _tokens(case):
    """Tokens that attention sees."""
    n = case["T"] * case["Hg"] * case["Wg"]
    return n if case["keep"] >= 1.0 else max(1, round(n * case["keep"]))


def work(case):
    b, h, d, bs = case["B"], case["H"], case["d"], case["block"]
    n, m = case["T"] * case["Hg"] * case["Wg"], _tokens(case)
    nb = -(-m // bs)
    kept = m if case["form"] == "dense" else min(min(case["k"], nb) * bs, m)
    flops = 4.0 * b * h * m * kept * d                              # the two products over the kept keys
    if case["form"] != "dense":
        flops += 2.0 * b * h * nb * nb * d                          # block scores
    if case["remainder"] >= 0:
        flops += 4.0 * b * h * m * (nb - min(case["k"], nb)) * d    # one mean key per dropped block
    if case["remainder"] == 1:                                      # C_J, A_I and A_I^T q
        flops += 4.0 * b * h * m * d * d + 2.0 * b * h * nb * (nb - min(case["k"], nb)) * d * d
    rows = 4.0 * b * h * m * d                                      # Q, K, V read and O written, at the tokens attended
    if case["prologue"]:
        rows += 2.0 * b * h * n * d                                 # the normalised, rotated Q and K are results too
    return {"bytes": 2.0 * rows, "flops": flops}


def tolerance(case):
    # bf16 probabilities, values and outputs with fp32 sums: against the fp32 CUDA-core kernel of the same contract the
    # outputs differ by 2.4e-3 .. 2.7e-3 (2-norm) and 0.011 .. 0.029 (largest); the routing is fp32 in a fixed order, so
    # only ties could move an index.  (The first-order term sums matrices that are themselves rounded to bf16.)
    return {"rel": 1e-2, "max": 0.2 if case["remainder"] == 1 else 0.12, "differ": 1e-3}


def _make(case, shape_n, gen, dev):
    """Q, K, V as the projection leaves them: unit normal values plus a per-frame and a per-window offset in Q and K."""
    b, h, d = case["B"], case["H"], case["d"]
    t, hg, wg = case["T"], case["Hg"], case["Wg"]
    if case["layout"] == "heads":
        q, k, v = (torch.empty(b, h, shape_n, d, dtype=torch.bfloat16, device=dev) for _ in range(3))
    elif case["layout"] == "tokens":
        q, k, v = (torch.empty(b, shape_n, h, d, dtype=torch.bfloat16, device=dev).transpose(1, 2) for _ in range(3))
    else:
        qkv = torch.empty(b, shape_n, 3, h, d, dtype=torch.bfloat16, device=dev)
        q, k, v = (qkv[:, :, i].transpose(1, 2) for i in range(3))
    tok = torch.arange(shape_n, device=dev)
    frame = tok // (hg * wg)
    window = (4 * ((tok // wg) % hg) // hg) * 4 + (4 * (tok % wg) // wg)
    by_frame = 0.5 * torch.randn(b, h, t, d, generator=gen, device=dev)
    by_window = 0.5 * torch.randn(b, h, 16, d, generator=gen, device=dev)
    for x in (q, k, v):
        for i in range(b):
            y = torch.randn(h, shape_n, d, generator=gen, device=dev)
            if x is not v:
                y += by_frame[i].index_select(1, frame)
                y += by_window[i].index_select(1, window)
                y *= case["qk_mult"]
            x[i].copy_(y)
    return q, k, v


def _like_bytes(x):
    return torch.zeros_like(x, dtype=torch.uint8)                   # (keeps the strides: codes are laid out as their tensor)


class State:
    pass


def prepare(case, seed):
    dev = torch.device("cuda")
    gen = torch.Generator(device=dev)
    gen.manual_seed(seed)
    s, w = State(), _workload(case)
    s.case = case
    b, h, d, bs = case["B"], case["H"], case["d"], case["block"]
    n, m = w.N, _tokens(case)
    s.q, s.k, s.v = _make(case, n, gen, dev)
    frame_blocks = w.blocks_per_frame if case["window"] else 0
    s.select = sva.make_select(case["mode"], case["k"], case["tau"], w.win_t, w.win_s, frame_blocks)
    s.status = torch.zeros(1, dtype=torch.int32, device=dev)
    if case["form"] == "attend":
        s.attend = sparse_attend(s.select, bs, s.status)
        return s

    # what attention reads: the tensors themselves, or the gathered subset
    s.aq, s.ak, s.av = s.q, s.k, s.v
    if case["keep"] < 1.0:
        pick = [torch.randperm(n, generator=gen, device=dev)[:m].sort().values for _ in range(b)]
        s.token_idx = torch.stack(pick).to(torch.int32)
        s.aq, s.ak, s.av = (torch.empty(b, h, m, d, dtype=torch.bfloat16, device=dev) for _ in range(3))
        s.result = torch.zeros_like(s.v)                            # the rows that are not attended keep what they held
    if case["prologue"]:
        s.gq, s.gk, s.cos, s.sin = (x.to(dev) for x in make_prologue_inputs(w, seed))
        s.raw_problem = sva.make_problem(s.q, s.k, None, None, n, bs)
        s.aq, s.ak = torch.empty_like(s.q), torch.empty_like(s.k)
        s.q_mean = torch.empty(b, h, w.Nb, d, dtype=torch.float32, device=dev)
        s.k_mean = torch.empty_like(s.q_mean)
    s.o = torch.zeros_like(s.av)
    nb = -(-m // bs)
    s.problem = sva.make_problem(s.aq, s.ak, s.av, s.o, m, bs)      # as bf16: routing, quantising, bf16 attention
    s.attn_problem = s.problem
    s.q_scale = s.k_scale = None
    if case["qk"] == "fp8":
        s.q8, s.k8 = _like_bytes(s.aq), _like_bytes(s.ak)
        s.q_scale = torch.zeros(b, h, nb, dtype=torch.float32, device=dev)
        s.k_scale = torch.zeros_like(s.q_scale)
        s.attn_problem = sva.make_problem(s.q8, s.k8, s.av, s.o, m, bs, 0.0, True)
        if case["smooth"]:
            s.key_mean = torch.zeros(b, h, d, dtype=torch.float32, device=dev)
            s.lse_shift = torch.zeros(b, h, m, dtype=torch.float32, device=dev)
            s.smooth_ws = torch.empty(sva.smooth_workspace_bytes(s.problem), dtype=torch.uint8, device=dev)
    elif case["qk"] == "fp4":
        s.q4, s.k4 = (torch.zeros(b * h, nb * 128, 64, dtype=torch.uint8, device=dev) for _ in range(2))
        s.q_sf, s.k_sf = (torch.zeros(b * h, nb, 1024, dtype=torch.uint8, device=dev) for _ in range(2))
        s.q_g, s.k_g = (torch.zeros(b * h, dtype=torch.float32, device=dev) for _ in range(2))
        s.quant_ws = torch.empty(max(256, 8 * b * h), dtype=torch.uint8, device=dev)
    if case["remainder"] >= 0:
        attn_bytes = sva.attn_remainder_workspace_bytes(s.problem, case["remainder"])
    elif case["qk"] == "fp4":
        attn_bytes = 256
    else:
        attn_bytes = sva.attn_one_call_workspace_bytes(s.attn_problem)
    s.attn_ws = torch.empty(max(256, attn_bytes), dtype=torch.uint8, device=dev)
    s.scores = None
    if case["remainder"] == 1:
        s.scores = torch.zeros(b, h, nb, nb, dtype=torch.float32, device=dev)
    if case["form"] == "sparse":
        s.select_ws = torch.empty(max(256, sva.select_workspace_bytes(s.attn_problem, s.select)), dtype=torch.uint8, device=dev)
        s.row_ptr = torch.zeros(b * h * nb + 1, dtype=torch.int32, device=dev)
        s.col_idx = torch.zeros(sva.select_max_nnz(s.attn_problem, s.select), dtype=torch.int32, device=dev)
    return s


def run(s):
    case = s.case
    if case["form"] == "attend":
        return {"o": s.attend(s.q, s.k, s.v), "status": s.status}
    if case["keep"] < 1.0:
        sva.gather_tokens(s.q, s.token_idx, s.aq, s.status)
        sva.gather_tokens(s.k, s.token_idx, s.ak, s.status)
        sva.gather_tokens(s.v, s.token_idx, s.av, s.status)
    q, k = s.aq, s.ak
    fp8 = case["qk"] == "fp8"
    if case["prologue"]:
        codes = (s.q8, s.k8, s.q_scale, s.k_scale) if fp8 else ()
        sva.qk_norm_rope_pool(s.raw_problem, s.q, s.k, s.gq, s.gk, s.cos, s.sin, 1e-6, q, k, s.q_mean, s.k_mean, *codes)
    elif fp8 and case["smooth"]:
        sva.quantize_qk_fp8_smooth_k(s.problem, q, k, s.q8, s.k8, s.q_scale, s.k_scale, s.key_mean, s.lse_shift, s.smooth_ws)
    elif fp8:
        sva.quantize_qk_fp8(s.problem, q, k, s.q8, s.k8, s.q_scale, s.k_scale)
    if fp8:
        q, k = s.q8, s.k8

    if case["form"] == "dense":
        sva.dense_attn_fwd(s.attn_problem, q, k, s.av, s.o, None, s.status, s.q_scale, s.k_scale, workspace=s.attn_ws)
        return {"o": s.o, "status": s.status}
    if case["prologue"]:
        sva.block_select_pooled(s.attn_problem, s.select, s.q_mean, s.k_mean, s.row_ptr, s.col_idx, s.select_ws, s.scores)
    else:
        sva.block_select(s.attn_problem, s.select, q, k, s.row_ptr, s.col_idx, s.select_ws, s.q_scale, s.k_scale, s.scores)

    if case["qk"] == "fp4":
        sva.quantize_qk_fp4(s.problem, q, k, s.q4, s.k4, s.q_sf, s.k_sf, s.q_g, s.k_g, s.quant_ws)
        sva.block_sparse_attn_fwd_fp4(s.problem, s.q4, s.k4, s.q_sf, s.k_sf, s.q_g, s.k_g, s.av, s.row_ptr, s.col_idx, s.o,
                                      None, s.status, s.attn_ws)
    elif case["remainder"] >= 0:
        sva.block_sparse_attn_remainder_fwd(s.problem, q, k, s.av, s.row_ptr, s.col_idx, s.o, None, s.status, case["remainder"],
                                            s.attn_ws, s.scores)
    else:
        sva.block_sparse_attn_fwd(s.attn_problem, q, k, s.av, s.row_ptr, s.col_idx, s.o, None, s.status, s.q_scale, s.k_scale,
                                  workspace=s.attn_ws)
    out = {"o": s.o, "row_ptr": s.row_ptr, "col_idx": s.col_idx, "status": s.status}
    if case["prologue"]:
        out["q"], out["k"] = s.aq, s.ak
    if case["smooth"]:
        out["lse_shift"] = s.lse_shift
    if case["keep"] < 1.0:
        sva.scatter_tokens(s.o, s.token_idx, s.result, s.status)
        out["o"] = s.result
    return out


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: sizes over the whole range (tokens 1 000 .. 48 000, 2 .. 32 heads), every option."""
    limit = 0.8 * work(_from_workload("xl", "xl"))["flops"]
    while True:
        c = dict(BASE)
        c["B"] = rng.choice((1, 1, 1, 2))
        c["H"] = _log_int(rng, 2, 32)
        c["block"] = rng.choice((128, 128, 64))
        per = [rng.randint(16, 48), rng.randint(16, 52)]
        if rng.random() < 0.3:                                      # frames of whole blocks: what the forced window needs
            per = [16 * rng.randint(1, 3), 16 * rng.randint(1, 3)]
        c["Hg"], c["Wg"] = per
        c["T"] = max(1, round(_log_int(rng, 1000, 48000) / (per[0] * per[1])))
        kind = rng.choice(("sparse", "sparse", "sparse", "sparse", "fp8", "fp8", "fp4", "remainder", "remainder", "dense", "pruned",
                           "attend"))
        if kind == "fp8":
            c.update(qk="fp8", prologue=rng.random() < 0.4)
            c["smooth"] = not c["prologue"] and rng.random() < 0.4
        elif kind == "fp4":
            c.update(qk="fp4", block=128, prologue=rng.random() < 0.5)
        elif kind == "remainder":
            c["remainder"] = rng.choice((0, 0, 1))
        elif kind == "pruned":
            c["keep"] = rng.choice((0.5, rng.uniform(0.3, 0.8)))
        elif kind in ("dense", "attend"):
            c["form"] = kind
        elif rng.random() < 0.3:
            c["prologue"] = True
        if kind in ("sparse", "fp8", "dense") and rng.random() < 0.15:
            c["d"] = 64
        layouts = ["heads", "heads", "tokens"]
        if c["qk"] == "bf16" and not c["prologue"]:
            layouts.append("packed")
        c["layout"] = rng.choice(layouts)
        c["qk_mult"] = rng.choice((1.0, 1.0, 1.5))
        nb = -(-_tokens(c) // c["block"])
        c["k"] = max(1, round(nb * rng.uniform(0.08, 0.3)))
        if rng.random() < 0.5:
            c.update(mode=1, tau=round(rng.uniform(0.8, 0.95), 3))
        if c["Hg"] * c["Wg"] % c["block"] == 0 and c["keep"] >= 1.0 and rng.random() < 0.6:
            c["window"] = True
        if nb < 4 or (c["window"] and c["k"] < 9):
            continue
        w = work(c)
        if w["flops"] <= limit and (c["remainder"] < 1 or c["B"] * c["H"] * nb <= 16000):
            return c
