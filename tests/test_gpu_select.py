"""Selection parity through the C ABI: kept sets bit-exact against the fp64 oracle (rows that
differ must be oracle near-ties, which are counted), CSR well-formed, scores within fp32 error."""
import numpy as np
import pytest
import torch

import _util as U
from paper_2606_23743_b200 import binding as B
from paper_2606_23743_b200.workloads import WORKLOADS, shrink

pytestmark = pytest.mark.gpu

CASES = {
    "tiny": WORKLOADS["tiny"],
    "medium": WORKLOADS["medium"],
    "ragged_tail": shrink(WORKLOADS["medium"], H=3, T=2, Hg=30, Wg=31, k=5),        # N = 1860
    "mass": shrink(WORKLOADS["large"], H=4, T=8),                                    # cap binds
    "mass_ragged_rows": shrink(WORKLOADS["large_ragged"], H=4, T=8),                 # variable counts
    "window": shrink(WORKLOADS["xl"], B=2, H=2, T=6),                                # 3x3 forced, k=37
    "window_gt_k": shrink(WORKLOADS["xl"], B=1, H=2, T=4, k=5),                      # |F| up to 9 > k
    "window_mass": shrink(WORKLOADS["xl"], B=1, H=2, T=4, mode=1, k=20, tau=0.5),
    "window_gt_k_72_blocks": shrink(WORKLOADS["xl"], B=1, H=2, T=6, k=5),
    "window_mass_72_blocks": shrink(WORKLOADS["xl"], B=1, H=2, T=6, mode=1, k=20, tau=0.5),
    "window_mass_204_blocks": shrink(WORKLOADS["xl"], B=1, H=1, T=17, mode=1, k=60, tau=0.7),
    "block64_d128": shrink(WORKLOADS["medium"], H=2, T=2, block=64, k=8),
    "k_ge_nb": shrink(WORKLOADS["tiny"], k=99),
    "k1": shrink(WORKLOADS["medium"], H=2, T=2, k=1),
}


@pytest.mark.parametrize("name", list(CASES))
def test_selection_matches_oracle(name):
    w = CASES[name]
    (q, k, _), (qb, kb, _) = U.host_inputs(w)
    rp, ci, sc = U.gpu_select(w, U.dev(q), U.dev(k), want_scores=True)
    sel, s_ref = U.oracle_select(w, qb, kb)
    assert np.abs(sc.cpu().numpy() - s_ref).max() < 2e-5
    assert int(rp[-1]) == ci.numel()
    n_diff, n_near = U.compare_selection(sel, rp, ci)
    print(f"{name}: rows {w.R} differing {n_diff} near-tie rows {n_near}")
    assert n_diff <= n_near


def test_exact_ties_resolve_to_lower_index():
    """Blocks with identical tokens give exactly equal scores on the GPU too."""
    w = shrink(WORKLOADS["medium"], H=1, T=2, k=3)        # Nb = 16
    g = torch.Generator().manual_seed(1)
    base = torch.randint(-2, 3, (4, w.d), generator=g).float()
    pat = torch.tensor([0, 1, 2, 3, 0, 1, 2, 3, 3, 2, 1, 0, 0, 0, 1, 1])
    x = base[pat].repeat_interleave(w.block, 0)[None, None].bfloat16().contiguous()
    rp, ci, sc = U.gpu_select(w, U.dev(x), U.dev(x), want_scores=True)
    bits = x.view(torch.int16).numpy().view(np.uint16)
    sel, s_ref = U.oracle_select(w, bits, bits)
    assert (sel.score_gap == 0).any()                     # the case really has boundary ties
    g = sc.cpu().numpy()
    np.testing.assert_allclose(g, s_ref, rtol=1e-6)
    assert g[0, 0, 0, 0] == g[0, 0, 0, 4] == g[0, 0, 0, 11]     # equal blocks score exactly equal
    np.testing.assert_array_equal(ci.cpu().numpy(), sel.col_idx)


def test_strided_views_and_determinism():
    w = shrink(WORKLOADS["medium"], H=2, T=2)
    (q, k, _), (qb, kb, _) = U.host_inputs(w)
    qkv = torch.zeros(w.B, w.n_alloc, 2, w.H, w.d, dtype=torch.bfloat16, device="cuda")   # packed [B,N,2,H,d]
    qkv[:, :, 0] = U.dev(q).permute(0, 2, 1, 3)
    qkv[:, :, 1] = U.dev(k).permute(0, 2, 1, 3)
    qv, kv = qkv[:, :, 0].permute(0, 2, 1, 3), qkv[:, :, 1].permute(0, 2, 1, 3)
    assert not qv.is_contiguous()
    rp1, ci1, _ = U.gpu_select(w, qv, kv)
    rp2, ci2, _ = U.gpu_select(w, U.dev(q), U.dev(k))
    assert torch.equal(rp1, rp2) and torch.equal(ci1, ci2)
    rp3, ci3, _ = U.gpu_select(w, qv, kv)
    assert torch.equal(ci1, ci3)


def test_workspace_too_small_is_rejected():
    w = CASES["mass"]
    (q, k, _), _ = U.host_inputs(w)
    qd, kd = U.dev(q), U.dev(k)
    p = B.make_problem(qd, kd, None, None, w.N, w.block)
    s = B.make_select(w.mode, w.k, w.tau)
    ws = torch.empty(B.select_workspace_bytes(p, s) - 256, dtype=torch.uint8, device="cuda")
    rp = torch.zeros(w.R + 1, dtype=torch.int32, device="cuda")
    ci = torch.zeros(B.select_max_nnz(p, s), dtype=torch.int32, device="cuda")
    with pytest.raises(B.SvaError) as e:
        B.block_select(p, s, qd, kd, rp, ci, ws)
    assert e.value.status == 3


@pytest.mark.parametrize("name", ["medium", "large_fp8"])
def test_routing_in_two_calls_equals_the_one_call(name):
    """sva_pool_qk + sva_block_select_pooled = sva_block_select (bf16 and e4m3 inputs); the means against
    the oracle's pooling."""
    import oracle
    from paper_2606_23743_b200 import binding as B
    from paper_2606_23743_b200.workloads import shrink
    w = shrink(WORKLOADS[name], H=2, T=3)
    (q, k, _), (qb, kb, _) = U.host_inputs(w)
    qd, kd = U.dev(q), U.dev(k)
    qs = ks = None
    if w.fp8:
        q8 = torch.zeros(qd.shape, dtype=torch.uint8, device="cuda"); k8 = torch.zeros_like(q8)
        qs = torch.zeros(w.B, w.H, w.Nb, dtype=torch.float32, device="cuda"); ks = torch.zeros_like(qs)
        B.quantize_qk_fp8(B.make_problem(qd, kd, None, None, w.N, w.block), qd, kd, q8, k8, qs, ks)
        qd, kd = q8, k8
    rp1, ci1, _ = U.gpu_select(w, qd, kd, q_scale=qs, k_scale=ks, fp8=w.fp8)
    p = B.make_problem(qd, kd, None, None, w.N, w.block, 0.0, w.fp8)
    s = B.make_select(w.mode, w.k, w.tau, w.win_t, w.win_s, w.blocks_per_frame if w.win_t >= 0 else 0)
    qm = torch.full((w.B, w.H, w.Nb, w.d), 7.0, dtype=torch.float32, device="cuda"); km = torch.full_like(qm, 7.0)
    B.pool_qk(p, qd, kd, qm, km, qs, ks)
    rp2 = torch.zeros(w.R + 1, dtype=torch.int32, device="cuda")
    ci2 = torch.zeros(B.select_max_nnz(p, s), dtype=torch.int32, device="cuda")
    ws = torch.empty(B.select_workspace_bytes(p, s), dtype=torch.uint8, device="cuda")
    B.block_select_pooled(p, s, qm, km, rp2, ci2, ws)
    torch.cuda.synchronize()
    assert torch.equal(rp1, rp2) and torch.equal(ci1, ci2[: int(rp2[-1])])
    if w.fp8:
        qb, kb = U.oracle_fp8_inputs(w, qb, kb, qd, kd, qs, ks)
    np.testing.assert_allclose(qm.cpu().numpy(), oracle.pool(qb, w.N, w.block), rtol=2e-6, atol=2e-7)
    np.testing.assert_allclose(km.cpu().numpy(), oracle.pool(kb, w.N, w.block), rtol=2e-6, atol=2e-7)


@pytest.mark.parametrize("T,Hg,Wg,mode,k,tau,d", [(25, 40, 40, 0, 20, 1.0, 128), (16, 64, 64, 1, 30, 0.95, 64)])
def test_many_blocks_per_head(T, Hg, Wg, mode, k, tau, d):
    """625 and 1024 (the maximum) 64-token blocks per head: every lane of the selection warp holds up to 32
    scores of its row; routing against the oracle, attention on sampled rows."""
    w = shrink(WORKLOADS["medium"], B=1, H=1, T=T, Hg=Hg, Wg=Wg, block=64, mode=mode, k=k, tau=tau, d=d, win_t=-1, win_s=-1)
    (q, kk, v), (qb, kb, vb) = U.host_inputs(w, seed=5)
    qd, kd, vd = U.dev(q), U.dev(kk), U.dev(v)
    rp, ci, sc = U.gpu_select(w, qd, kd, want_scores=True)
    sel, s_ref = U.oracle_select(w, qb, kb)
    assert np.abs(sc.cpu().numpy() - s_ref).max() < 2e-5
    n_diff, n_near = U.compare_selection(sel, rp, ci)
    assert n_diff <= n_near
    o, lse, st = U.gpu_attn(w, qd, kd, vd, rp, ci)
    assert st == 0
    U.check_attn_vs_oracle(w, qb, kb, vb, rp, ci, o, lse, U.sample_rows(w.R, w.Nb, 6))


def _rule(scores, mode, k, tau):
    """The routing rule, one candidate at a time (float64 masses); the smallest distance of the mass from tau on the way."""
    order = sorted((j for j in range(len(scores)) if not np.isnan(scores[j])), key=lambda j: (-scores[j], j))
    x = scores.astype(np.float64)
    e = np.exp(x - x[order[0]]) if mode == 1 else None
    z = e[order].sum() if mode == 1 else 1.0
    kept, mass, margin = [], 0.0, np.inf
    for j in order[:k]:
        kept.append(j)
        if mode == 1:
            mass += e[j] / z
            margin = min(margin, abs(mass - tau))
            if mass >= tau:
                break
    return sorted(kept), margin


@pytest.mark.parametrize("nb", [1, 2, 31, 33, 128, 129, 257, 385, 513, 1024])
@pytest.mark.parametrize("mode", [0, 1])
def test_threshold_search_on_awkward_scores(nb, mode):
    """Rows whose scores are equal, nearly equal, far apart, infinite or a few values many times: the search for the
    threshold must end and keep what the rule keeps (scores are made exact: one non-zero dimension)."""
    rng = np.random.default_rng(nb)
    kinds = [rng.standard_normal(nb), np.zeros(nb), 1.0 + 2.0 ** -22 * rng.integers(0, 3, nb), rng.integers(-2, 3, nb) * 1.0,
             -np.exp(rng.standard_normal(nb) * 4.0), np.linspace(-3.0, 3.0, nb)]
    if mode == 0:
        wild = rng.standard_normal(nb)
        wild[rng.integers(0, nb, 2)] = (np.inf, -np.inf)
        kinds += [rng.standard_normal(nb) * 10.0 ** rng.integers(-30, 30, nb), wild, 1e-40 * rng.standard_normal(nb)]
    H, d = len(kinds), 128
    n = nb * 128
    kbar = np.zeros((1, H, nb, d), np.float32)
    for h, x in enumerate(kinds):
        kbar[0, h, :, 0] = x
    qbar = np.zeros_like(kbar)
    qbar[..., 0] = 1.0
    t = torch.empty(1, H, n, d, dtype=torch.bfloat16, device="cuda")
    p = B.make_problem(t, t, None, None, n, 128, 1.0)
    for k in sorted({1, max(1, nb // 10), max(1, nb // 2), nb}):
        s = B.make_select(mode, k, 0.87)
        ws = torch.empty(max(B.select_workspace_bytes(p, s), 256), dtype=torch.uint8, device="cuda")
        rp = torch.zeros(H * nb + 1, dtype=torch.int32, device="cuda")
        ci = torch.zeros(B.select_max_nnz(p, s), dtype=torch.int32, device="cuda")
        B.block_select_pooled(p, s, torch.tensor(qbar).cuda(), torch.tensor(kbar).cuda(), rp, ci, ws)
        rp, ci = rp.cpu().numpy(), ci.cpu().numpy()
        for h in range(H):
            want, margin = _rule(kbar[0, h, :, 0], mode, k, 0.87)
            if margin < 1e-5:                                 # fixed-point masses (2^-31 each) against float64
                continue
            for r in (h * nb, h * nb + nb - 1):
                assert ci[rp[r]:rp[r + 1]].tolist() == want, (h, k)


@pytest.mark.parametrize("nb,k,window", [(16, 4, False), (16, 16, False), (40, 33, False), (129, 70, False), (16, 9, True), (68, 9, True),
                                         (132, 20, True)])
def test_rows_of_a_known_length_are_written_whole(nb, k, window):
    """A NaN score is never selected, so a row of top-k can find fewer than the k blocks its row_ptr covers: the entries left
    over are block 0, whatever col_idx held before."""
    d, n = 128, nb * 128
    rng = np.random.default_rng(nb)
    qbar, kbar = (rng.standard_normal((1, 3, nb, d)).astype(np.float32) for _ in range(2))
    qbar[0, 0, [0, nb // 2, nb - 1]] = np.nan                    # head 0: rows without a candidate
    kbar[0, 1, [1, nb - 1]] = np.nan                             # head 1: two blocks that no row can pick; head 2: as usual
    t = torch.empty(1, 3, n, d, dtype=torch.bfloat16, device="cuda")
    p = B.make_problem(t, t, None, None, n, 128)
    s = B.make_select(0, k, 1.0, 1, 1, 4) if window else B.make_select(0, k)
    ws = torch.empty(max(B.select_workspace_bytes(p, s), 256), dtype=torch.uint8, device="cuda")
    got = []
    for junk in (-7, 0x7fffffff):
        rp = torch.full((3 * nb + 1,), junk, dtype=torch.int32, device="cuda")
        ci = torch.full((B.select_max_nnz(p, s),), junk, dtype=torch.int32, device="cuda")
        B.block_select_pooled(p, s, torch.tensor(qbar).cuda(), torch.tensor(kbar).cuda(), rp, ci, ws)
        got.append((rp.cpu().numpy(), ci.cpu().numpy().reshape(3 * nb, k)))
    rp, ci = got[0]
    assert np.array_equal(rp, np.arange(3 * nb + 1) * k) and np.array_equal(rp, got[1][0]) and np.array_equal(ci, got[1][1])
    scores = np.einsum("hid,hjd->hij", qbar[0], kbar[0]) / np.sqrt(np.float32(d))
    for h in range(3):
        for i in range(nb):
            x = scores[h, i].astype(np.float64)
            forced = [j for j in range(nb) if window and abs(i // 4 - j // 4) <= 1 and abs(i % 4 - j % 4) <= 1]
            real = [j for j in range(nb) if not np.isnan(x[j]) and j not in forced]
            kept = sorted(forced + sorted(real, key=lambda j: (-x[j], j))[:k - len(forced)])
            assert ci[h * nb + i].tolist() == kept + [0] * (k - len(kept)), (h, i)


@pytest.mark.parametrize("B_,H,Nb,block,d,fp8,mode,k,window,layout,values", [
    (1, 1, 1, 128, 128, False, 0, 1, False, "heads", "normal"),           # one launch: one block, ragged
    (1, 3, 9, 128, 128, False, 1, 4, False, "tokens", "normal"),          # ... CTAs of the cluster without a block
    (2, 7, 16, 64, 64, True, 0, 5, True, "heads", "normal"),              # ... 14 heads, the most blocks, e4m3, forced window
    (1, 4, 12, 64, 128, False, 0, 9, False, "heads", "nan"),              # ... rows of NaN scores come out short
    (1, 2, 13, 128, 64, True, 1, 40, False, "packed8", "zero"),           # ... every score equal, k beyond Nb
    (1, 15, 16, 64, 64, False, 0, 5, False, "heads", "normal"),           # means, then scores and selection: one head too many
    (2, 7, 64, 64, 128, False, 0, 11, False, "packed", "normal"),         # ... the most blocks
    (1, 12, 44, 128, 64, False, 1, 12, True, "heads", "normal"),          # ... forced window and mass
    (1, 8, 44, 64, 64, False, 0, 3, True, "tokens", "ties"),              # ... window larger than k, equal scores
    (1, 2, 31, 128, 128, False, 1, 40, False, "heads", "zero"),
    (1, 4, 20, 64, 128, False, 0, 7, False, "heads", "nan"),
    (1, 9, 33, 64, 128, True, 1, 6, False, "tokens", "normal"),           # ... e4m3 codes, a row in a CTA of its own
    (2, 9, 64, 128, 128, False, 1, 9, False, "packed", "normal"),
    (1, 24, 17, 128, 128, False, 0, 2, False, "heads", "ties"),
    (1, 5, 65, 64, 64, False, 1, 9, False, "heads", "normal"),            # the general kernels, one block more
    (1, 4, 68, 64, 64, False, 1, 12, True, "heads", "normal"),            # ... forced window and mass
    (1, 3, 72, 128, 128, True, 1, 40, True, "tokens", "normal"),
    (2, 3, 132, 64, 128, False, 0, 3, True, "tokens", "ties"),            # ... window larger than k, equal scores
    (1, 4, 68, 64, 128, False, 0, 12, True, "heads", "nan"),              # ... forced window, rows of NaN scores come out short
    (1, 4, 132, 64, 64, False, 1, 12, True, "packed", "nan"),
    (1, 2, 100, 64, 64, False, 1, 150, True, "heads", "zero"),
])
def test_routing_of_small_problems(B_, H, Nb, block, d, fp8, mode, k, window, layout, values):
    """Few blocks per head take kernels of their own (the last rows are of the general ones), which rank a row's candidates instead of searching a threshold: the lists are what the sequential
    rule takes from the kernel's own scores, and routing in one call is routing from means that another call has made, byte for byte."""
    N = Nb * block - (37 if Nb % 2 else 0)
    g = torch.Generator(device="cuda").manual_seed(Nb)
    shape = {"heads": (2, B_, H, N, d), "tokens": (2, B_, N, H, d)}.get(layout, (B_, N, 2, H, d))
    x = torch.randn(shape, generator=g, device="cuda")
    qk = x.transpose(2, 3) if layout == "tokens" else x if layout == "heads" else x.permute(2, 0, 3, 1, 4)       # [2, B, H, N, d] views
    if values == "ties":
        qk[:, :, :, block:] = qk[:, :, :, :1]                             # all blocks but the first alike
    elif values == "zero":
        qk.zero_()
    elif values == "nan":
        qk[1, :, 1, : 3 * block] = float("nan")                           # keys of three blocks: no candidates
        qk[0, :, 2, :5] = float("nan")                                    # a query block without a score
        qk[1, :, 3, 7] = float("inf")
    scales = [None, None]
    if fp8:
        qk = qk.to(torch.float8_e4m3fn).view(torch.uint8)
        scales = [torch.rand(B_, H, Nb, generator=g, device="cuda") + 0.5 for _ in range(2)]
    else:
        qk = qk.to(torch.bfloat16)
    q, kk = qk[0], qk[1]
    tau, bpf = 0.7, 4
    p = B.make_problem(q, kk, None, None, N, block, 0.0, True) if fp8 else B.make_problem(q, kk, None, None, N, block)
    s = B.make_select(mode, k, tau, *((1, 1, bpf) if window else (-1, -1, 0)))
    got = []
    for split in (False, True):
        ws = torch.full((B.select_workspace_bytes(p, s),), 255, dtype=torch.uint8, device="cuda")
        rp = torch.full((B_ * H * Nb + 1,), -7, dtype=torch.int32, device="cuda")
        ci = torch.full((B.select_max_nnz(p, s),), -7, dtype=torch.int32, device="cuda")
        sc = torch.full((B_, H, Nb, Nb), -7.0, device="cuda")
        if split:
            qm, km = (torch.zeros(B_, H, Nb, d, device="cuda") for _ in range(2))
            B.pool_qk(p, q, kk, qm, km, *scales)
            B.block_select_pooled(p, s, qm, km, rp, ci, ws, sc)
        else:
            B.block_select(p, s, q, kk, rp, ci, ws, *scales, sc)
        torch.cuda.synchronize()
        got.append((rp, ci, sc.view(torch.int32)))
    for a, b in zip(*got):
        assert torch.equal(a, b)
    rp, ci, sc = got[0][0].cpu().numpy(), got[0][1].cpu().numpy(), got[0][2].view(torch.float32).cpu().numpy().reshape(-1, Nb)
    for r in range(B_ * H * Nb):
        v, I = sc[r].astype(np.float64), r % Nb
        kept = [J for J in range(Nb) if window and abs(I // bpf - J // bpf) <= 1 and abs(I % bpf - J % bpf) <= 1]
        cand = np.flatnonzero(~np.isnan(v))
        w = np.zeros(Nb)
        if cand.size:
            with np.errstate(invalid="ignore"):
                w[cand] = np.exp(v[cand] - v[cand].max())
            w /= w.sum()
        near = False                                                      # (the mass comes within summation noise of tau: either is right)
        for J in sorted((c for c in cand if c not in kept), key=lambda c: (-v[c], c)):
            mass = w[kept].sum()
            near = near or (mode == 1 and kept and abs(mass - tau) < 1e-5)
            if len(kept) >= min(k, Nb) or (mode == 1 and kept and mass >= tau):
                break
            kept.append(J)
        want = sorted(kept)
        if mode == 0 and (not window or k >= 9):                          # (a row's count is known: no window larger than k)
            want += [0] * (min(k, Nb) - len(want))                        # (a short row is filled up)
        have = ci[rp[r]:rp[r + 1]].tolist()
        if values == "nan":
            have, want = sorted(have), sorted(want)
        assert near or have == want, (r, have, want)


@pytest.mark.parametrize("mode,k,window,H,Nb,by_rank", [
    (mode, k, window, H, Nb, by_rank) for mode, k, window, lines in [
        (0, 9, False, ((160, 64), (310, 44))), (0, 5, True, ((160, 64), (310, 44))),
        (1, 12, False, ((187, 64), (363, 44))), (1, 30, True, ((187, 64), (363, 44)))]
    for H, Nb, by_rank in [(lines[0][0], 64, True), (lines[0][0] + 1, 64, False), (500, 64, False),
                           (lines[1][0], 44, True), (lines[1][0] + 1, 44, False), (900, 40, True)]])
def test_heads_at_the_end_of_counting_ranks(mode, k, window, H, Nb, by_rank):
    """Many heads of 41 to 64 blocks search a threshold in a kernel of its own (which leaves the scores in the workspace), fewer count
    ranks: on either side of the line a call returns what calls on a few of its heads return."""
    g = torch.Generator(device="cuda").manual_seed(Nb)
    qm, km = (torch.randn(1, H, Nb, 64, generator=g, device="cuda") for _ in range(2))
    s = B.make_select(mode, k, 0.8, *((1, 1, 4) if window else (-1, -1, 0)))

    def route(h0, h1):
        t = torch.empty(1, h1 - h0, Nb * 64, 64, dtype=torch.bfloat16, device="cuda")
        p = B.make_problem(t, t, None, None, Nb * 64, 64)
        ws = torch.full((B.select_workspace_bytes(p, s),), 255, dtype=torch.uint8, device="cuda")
        rp = torch.full(((h1 - h0) * Nb + 1,), -7, dtype=torch.int32, device="cuda")
        ci = torch.full((B.select_max_nnz(p, s),), -7, dtype=torch.int32, device="cuda")
        B.block_select_pooled(p, s, qm[:, h0:h1].contiguous(), km[:, h0:h1].contiguous(), rp, ci, ws)
        torch.cuda.synchronize()
        scores = ws[ws.numel() - (4 * (h1 - h0) * Nb * Nb + 255) // 256 * 256:]
        return rp[1:] - rp[:-1], ci[:int(rp[-1])], bool((scores == 255).all())

    counts, blocks, untouched = route(0, H)
    assert untouched == by_rank
    parts = [route(h, min(h + 100, H)) for h in range(0, H, 100)]
    assert all(p[2] for p in parts)
    assert torch.equal(counts, torch.cat([p[0] for p in parts])) and torch.equal(blocks, torch.cat([p[1] for p in parts]))


@pytest.mark.parametrize("H,Nb,block,d,fp8", [(2, 16, 64, 64, False), (14, 16, 128, 128, False), (1, 1, 128, 128, False), (3, 9, 64, 128, True)])
@pytest.mark.parametrize("mode", [0, 1])
def test_small_problems_where_no_cluster_fits(H, Nb, block, d, fp8, mode):
    """A partition of the device can be too small for the clusters of the one-launch routing (the test switch asks for larger ones than
    exist): the call then takes other kernels and returns the same."""
    N = Nb * block - 5
    g = torch.Generator(device="cuda").manual_seed(Nb)
    q, k = torch.randn(2, 1, H, N, d, generator=g, device="cuda").to(torch.bfloat16)
    scales = [None, None]
    if fp8:
        q, k = (x.to(torch.float8_e4m3fn).view(torch.uint8) for x in (q, k))
        scales = [torch.rand(1, H, Nb, generator=g, device="cuda") + 0.5 for _ in range(2)]
    p, s = B.make_problem(q, k, None, None, N, block, 0.0, fp8), B.make_select(mode, max(1, Nb // 3), 0.6)

    def route(entry):
        rp = torch.full((H * Nb + 1,), -7, dtype=torch.int32, device="cuda")
        ci = torch.full((B.select_max_nnz(p, s),), -7, dtype=torch.int32, device="cuda")
        sc = torch.full((1, H, Nb, Nb), -7.0, device="cuda")
        ws = torch.full((B.select_workspace_bytes(p, s),), 255, dtype=torch.uint8, device="cuda")
        entry(p, s, q, k, rp, ci, *((ws,) if entry is B.block_select else ()), *scales, sc)
        torch.cuda.synchronize()
        return rp, ci, sc

    want = route(B.block_select)
    try:
        B.debug_set_mode(64)
        got = [route(B.block_select), route(B.block_select_noalloc)]
    finally:
        B.debug_set_mode(0)
    for x in got + [route(B.block_select)]:
        assert all(torch.equal(a, b) for a, b in zip(want, x))


@pytest.mark.parametrize("d,block,fp8", [(64, 64, True), (128, 64, True), (64, 128, True), (128, 128, True), (64, 64, False), (128, 64, False),
                                         (64, 128, False), (128, 128, False)])
@pytest.mark.parametrize("run", [3, 0], ids=["run3", "longest"])
def test_pooling_in_runs_of_blocks(run, d, block, fp8):
    """A CTA pools a run of blocks, the longer the larger the call, up to 128 KB: the means are those of calls on one head each, which are
    small enough for a block per CTA, byte for byte, and those of another program."""
    block_bytes = block * d * (1 if fp8 else 2)
    blocks = (run or (128 << 10) // block_bytes) * ((16 << 20) // block_bytes)          # of Q and K together
    H = 40
    Nb = blocks // (2 * H) + 1
    Nb += Nb % max(run, 2) == 0                                             # (the last run of a head is a short one)
    N = Nb * block - 21
    g = torch.Generator(device="cuda").manual_seed(d + block)
    q, k = (torch.randn(1, N, H, d, generator=g, device="cuda", dtype=torch.bfloat16).transpose(1, 2) for _ in range(2))
    scales = [None, None]
    if fp8:
        q, k = (x.to(torch.float8_e4m3fn).view(torch.uint8) for x in (q, k))
        scales = [torch.rand(1, H, Nb, generator=g, device="cuda") + 0.5 for _ in range(2)]

    def pool(h0, h1):
        part = [x[:, h0:h1] for x in (q, k)]
        means = [torch.full((1, h1 - h0, Nb, d), float("nan"), device="cuda") for _ in range(2)]
        B.pool_qk(B.make_problem(*part, None, None, N, block, 0.0, fp8), *part, *means, *(s if s is None else s[:, h0:h1].contiguous() for s in scales))
        return torch.stack(means)

    got = pool(0, H)
    assert torch.equal(got, torch.cat([pool(h, h + 1) for h in range(H)], dim=2))
    h = H - 1
    for i, x in enumerate((q, k)):
        y = torch.zeros(Nb * block, d, dtype=torch.float64, device="cuda")
        y[:N] = (x[0, h].view(torch.float8_e4m3fn) if fp8 else x[0, h]).double()
        count = torch.full((Nb, 1), float(block), dtype=torch.float64, device="cuda")
        count[-1] = N - (Nb - 1) * block
        want = y.reshape(Nb, block, d).sum(1) / count
        if fp8:
            want *= scales[i][0, h].double()[:, None]
        # (sums of at most 128 values in fp32: each addition's error is below 2^-24 of a partial sum, and those stay below sum |y|)
        bound = 2.0 ** -24 * 130 * y.abs().reshape(Nb, block, d).sum(1) / count * (scales[i][0, h].double()[:, None] if fp8 else 1.0)
        assert ((got[i, 0, h].double() - want).abs() <= bound + 1e-30).all()
