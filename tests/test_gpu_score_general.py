"""The general score kernel where its launches change shape: key blocks at the limits of a cluster's shared memory (four heads: 1064 per CTA, 552
where twice the CTAs still run at once; fewer heads: 552 x 4 / heads), CTAs as many as SMs and one more, fp32 rows at the
limit of two CTAs per SM (472 blocks)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2409_12490_b200 import binding as cp
from paper_2409_12490_b200.inputs import make_uniform_qkv

from helpers import compare_scores, f32

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,d,g,n2,segments", [
    ("bf16", 128, 4, 552, 138), ("f16", 128, 4, 552, 184), ("bf16", 128, 4, 553, 93), ("f32", 128, 4, 553, 111),
    ("f16", 64, 4, 148, 148), ("bf16", 128, 4, 149, 149), ("f32", 64, 2, 1105, 79), ("bf16", 64, 1, 2209, 60),
    ("bf16", 128, 4, 553, 74), ("f32", 64, 4, 553, 79), ("bf16", 64, 4, 1064, 152), ("f16", 128, 4, 1065, 153), ("f32", 128, 4, 472, 158),
    ("f32", 128, 4, 473, 158), ("f32", 128, 1, 1889, 158), ("bf16", 128, 4, 1105, 12), ("f16", 64, 4, 2209, 6), ("bf16", 64, 4, 4417, 3), ("f16", 64, 4, 8191, 2),
])
def test_shapes_of_the_launch(dtype, d, g, n2, segments):
    r = -(-n2 // segments)
    n = 16 * n2 - 3
    Q, K, _ = make_uniform_qkv(1, g, 1, n, d, dtype=dtype, seed=n2)
    dt = {"bf16": torch.bfloat16, "f16": torch.float16, "f32": torch.float32}[dtype]
    prob = cp.Problem(1, g, 1, n, d, 16 * r, 16, r, dt)
    ws = cp.alloc_workspace(prob)
    S_prev_ref = oracle.estimate(K.expand(1, g, n, d), K, 16 * r, 16, est_scale=1.0)
    S = cp.estimate(prob, Q.cuda(), K.cuda(), ws, S_prev=torch.from_numpy(S_prev_ref).cuda())
    assert cp.device_status(ws) == 0
    compare_scores(S, oracle.estimate(Q, K, 16 * r, 16, est_scale=1.0, alpha=f32(0.25), S_prev=S_prev_ref))
