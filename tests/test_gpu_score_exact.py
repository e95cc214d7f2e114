"""Exact scores from byte products: sizes around its tiles of 32 blocks, row groups of 64 / (heads per CTA) segments and parts per CTA,
and representatives that do not fit 31 bits beside their row's largest (those are summed in fp64 instead)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2409_12490_b200 import binding as cp
from paper_2409_12490_b200.inputs import make_uniform_qkv

from helpers import compare_scores, f32

pytestmark = pytest.mark.gpu
DT = {"bf16": torch.bfloat16, "f16": torch.float16}


def check(Q, K, dtype, seg, blk, est_scale=1.0, fuse=False, atol=1e-9):
    B, Hq, n, d = Q.shape
    prob = cp.Problem(B, Hq, K.shape[1], n, d, seg, blk, max(seg // blk, 4), DT[dtype], est_scale=est_scale, flags=cp.FLAG_FORCE_SPLIT_SCORE)
    ws = cp.alloc_workspace(prob)
    S_prev = S_prev_ref = None
    if fuse:
        S_prev_ref = oracle.estimate(K.repeat_interleave(Hq // K.shape[1], 1), K, seg, blk, est_scale=f32(est_scale))
        S_prev = torch.from_numpy(S_prev_ref).cuda()
    S = cp.estimate(prob, Q.cuda(), K.cuda(), ws, S_prev=S_prev)
    assert cp.device_status(ws) == 0
    compare_scores(S, oracle.estimate(Q, K, seg, blk, est_scale=f32(est_scale), alpha=f32(0.25), S_prev=S_prev_ref), atol)


@pytest.mark.parametrize("dtype,B,Hkv,g,n,seg,blk", [
    ("bf16", 1, 1, 4, 31 * 16, 16, 16),        # one tile, one block short; more segments than a row group has
    ("f16", 1, 2, 4, 33 * 16 - 5, 32, 16),     # a tile and a block, odd rows
    ("bf16", 2, 1, 8, 1301, 128, 32),          # two subgroups of heads
    ("f16", 1, 3, 2, 2050, 64, 32),            # 32 segments and one more
    ("bf16", 1, 5, 1, 4097, 64, 64),           # 64 segments and one more
    ("bf16", 1, 8, 4, 6000, 256, 16),          # parts that begin inside a row group
    ("f16", 1, 1, 6, 900, 32, 32),
])
@pytest.mark.parametrize("fuse", [False, True])
def test_sizes(dtype, B, Hkv, g, n, seg, blk, fuse):
    Q, K, _ = make_uniform_qkv(B, Hkv * g, Hkv, n, 128, dtype=dtype, seed=n + g)
    check(Q, K, dtype, seg, blk, fuse=fuse)


@pytest.mark.parametrize("dtype", ["bf16", "f16"])
@pytest.mark.parametrize("where", ["blocks", "rows", "both", "outliers", "tiny", "scale"])
def test_values_that_do_not_fit(dtype, where):
    Q, K, _ = make_uniform_qkv(1, 8, 2, 1500, 128, dtype=dtype, seed=5)
    small = 3e-8 if dtype == "bf16" else 6e-8
    if where in ("blocks", "both"):
        K[:, :, 300:700, 7] = small              # whole blocks whose maximum and minimum are tiny in one channel
    if where in ("rows", "both"):
        Q[:, 1::2, 256:900, 100] = -small
    if where == "outliers":                      # fp16: beyond 2^6, where multiples of 2^-24 no longer fit
        Q[:, :, ::97, 3] = 80.0
        K[:, 0, ::53, 3] = -80.0
        Q[:, :, :, 4] = small
        K[:, :, :, 5] = small
    if where == "tiny":                          # whole rows near the bottom of the type
        Q *= 2e-38 if dtype == "bf16" else 1e-6
        K[:, 1] *= 0.0
    # sums of 128 products of up to 80 x 80 are good to 128 x 6400 x 2^-53 in the oracle
    check(Q, K, dtype, 128, 32, est_scale=0.0883 if where == "scale" else 1.0)
