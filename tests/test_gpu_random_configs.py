"""Seeded random small configurations (token grid, block size, head dimension, dtype, rule, window, dense):
routing and attention against the oracle, with the workspaces filled with NaN patterns beforehand."""
import numpy as np
import pytest
import torch

import _util as U
from paper_2606_23743_b200 import binding as B
from paper_2606_23743_b200.workloads import WORKLOADS, shrink

pytestmark = pytest.mark.gpu


def _case(rng, many=False):
    block = int(rng.choice([64, 128])); d = int(rng.choice([64, 128])); fp8 = bool(rng.integers(0, 2))
    T, Hg, Wg = int(rng.integers(1, 7)), int(rng.integers(1, 12)), int(rng.integers(1, 40))
    if many:                                                  # 65 to 224 blocks per head, every other time frames of whole blocks
        T = int(rng.integers(5, 9))
        Hg, Wg = (block, int(rng.integers(13, 29))) if rng.random() < 0.5 else (block // 2, int(rng.integers(27, 57)))
    N = T * Hg * Wg
    Nb = -(-N // block)
    kw = dict(B=int(rng.integers(1, 3)), H=int(rng.integers(1, 4)), T=T, Hg=Hg, Wg=Wg, block=block, d=d,
              mode=int(rng.integers(0, 2)), k=int(rng.integers(1, 12)), tau=float(rng.choice([0.5, 0.9, 0.99, 1.0])),
              fp8=fp8, sigma_f=float(rng.choice([0.3, 0.65, 1.0])), sigma_w=float(rng.choice([0.0, 0.5])),
              qk_mult=float(rng.choice([1.0, 1.5, 3.0])), win_t=-1, win_s=-1)
    if rng.random() < (0.7 if many else 0.25) and N % block == 0 and Nb % T == 0:
        kw.update(win_t=int(rng.integers(0, 2)), win_s=int(rng.integers(0, 2)))
    return shrink(WORKLOADS["medium"], **kw), rng.random() < 0.2


@pytest.mark.parametrize("seed", [1, 2, 3])
def test_random_configurations(seed):
    _run(seed, 40)


@pytest.mark.parametrize("seed", [4, 5])
def test_random_configurations_of_many_blocks(seed):
    """The same above 64 blocks per head, where scores and selection are kernels of their own."""
    _run(seed, 12, many=True)


def _run(seed, cases, many=False):
    rng = np.random.default_rng(seed)
    for case in range(cases):
        w, dense = _case(rng, many)
        what = f"seed {seed} case {case}: {w}"
        (q, k, v), (qb, kb, vb) = U.host_inputs(w, seed=1000 * seed + case)
        qd, kd, vd = U.dev(q), U.dev(k), U.dev(v)
        qs = ks = None
        if w.fp8:
            q8 = torch.zeros(qd.shape, dtype=torch.uint8, device="cuda"); k8 = torch.zeros_like(q8)
            qs = torch.zeros(w.B, w.H, w.Nb, dtype=torch.float32, device="cuda"); ks = torch.zeros_like(qs)
            B.quantize_qk_fp8(B.make_problem(qd, kd, None, None, w.N, w.block), qd, kd, q8, k8, qs, ks)
            torch.cuda.synchronize()
            qb, kb = U.oracle_fp8_inputs(w, qb, kb, q8, k8, qs, ks)
            qd, kd = q8, k8
        rp, ci, _ = U.gpu_select(w, qd, kd, q_scale=qs, k_scale=ks, fp8=w.fp8)
        sel, _ = U.oracle_select(w, qb, kb)
        n_diff, n_near = U.compare_selection(sel, rp, ci)
        assert n_diff <= n_near, what
        o, lse, st = U.gpu_attn(w, qd, kd, vd, rp, ci, dense=dense, q_scale=qs, k_scale=ks, fp8=w.fp8)
        assert st == 0, what
        rows = U.sample_rows(w.R, w.Nb, 8, seed=case)
        # peaked rows of these small cases return single V rows of magnitude up to ~4.5, where one bf16 unit is
        # 0.031: the absolute bound is the workloads' 2e-2 or one unit of the largest output, whichever is larger
        unit = 2.0 ** -7 * float(o[:, :, :w.N].float().abs().max())
        tol = dict(rel_tol=U.FP8_REL_L2, abs_tol=max(5e-2, unit)) if w.fp8 else dict(abs_tol=max(U.BF16_MAX_ABS, unit))
        U.check_attn_vs_oracle(w, qb, kb, vb, rp, ci, o, lse, rows, dense=dense, **tol)
        if w.n_alloc > w.N:
            assert (o[:, :, w.N:] == 7.0).all(), what
