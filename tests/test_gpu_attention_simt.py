"""The SIMT attention kernel against the fp64 oracle: both row-tile sizes, segments and blocks that are not multiples of its
tiles, ragged tails, and values that are not finite."""
import numpy as np
import pytest
import torch

import oracle
from paper_2409_12490_b200 import binding as cp
from paper_2409_12490_b200.inputs import make_uniform_qkv

from helpers import f32

pytestmark = pytest.mark.gpu

TDT = {"bf16": torch.bfloat16, "f16": torch.float16, "f32": torch.float32}


def assert_close(O, O_ref, V, dtype):
    """One rounding of O (unit roundoff u), fp32 arithmetic before it: logits, exponentials and sums over up to 2^11 keys are
    good to 2^-17 of max|V| together."""
    u = {"bf16": 2.0 ** -8, "f16": 2.0 ** -11, "f32": 2.0 ** -24}[dtype]
    err = np.abs(O.float().cpu().numpy().astype(np.float64) - O_ref)
    assert (err <= u * np.abs(O_ref) + 2.0 ** -17 * float(V.float().abs().max())).all(), float(err.max())


@pytest.mark.parametrize("dtype,d", [("f32", 64), ("f32", 128), ("bf16", 64), ("f16", 128)])
@pytest.mark.parametrize("B,Hq,Hkv,n,seg,blk,k", [
    (1, 1, 1, 1, 16, 16, 2), (1, 2, 1, 65, 64, 32, 3), (2, 2, 1, 331, 60, 20, 7), (1, 4, 2, 1024, 128, 32, 8),
    (2, 8, 2, 1339, 192, 48, 9), (1, 8, 8, 2400, 100, 4, 61)])
def test_sparse_and_dense_match_the_oracle(dtype, d, B, Hq, Hkv, n, seg, blk, k):
    Q, K, V = make_uniform_qkv(B, Hq, Hkv, n, d, dtype=dtype, seed=n)
    prob = cp.Problem(B, Hq, Hkv, n, d, seg, blk, k, TDT[dtype], flags=cp.FLAG_FORCE_SIMT)
    ws = cp.alloc_workspace(prob)
    Qd, Kd, Vd = Q.cuda(), K.cuda(), V.cuda()
    idx, cnt = cp.select(prob, cp.estimate(prob, Qd, Kd, ws), ws)
    O, lse = cp.attention(prob, Qd, Kd, Vd, idx, cnt, ws, want_lse=True)
    Od = cp.dense_attention(prob, Qd, Kd, Vd, ws)
    assert cp.device_status(ws) == 0
    sm = f32(1.0 / np.sqrt(d))
    O_ref, lse_ref = oracle.sparse_attention(Q, K, V, idx.cpu().numpy(), cnt.cpu().numpy(), seg, blk, sm)
    assert_close(O, O_ref, V, dtype)
    assert np.abs(lse.cpu().numpy() - lse_ref).max() <= 1e-4
    assert_close(Od, oracle.dense_attention(Q, K, V, sm)[0], V, dtype)


def test_segment_far_longer_than_the_sequence():
    """2^29 tokens to the segment: tiles are counted over the rows there are, not over the segment's (2^33 tiles for 512 heads)."""
    n, seg, H = 100, 1 << 29, 512
    Q, K, V = make_uniform_qkv(1, H, 1, n, 64, dtype="f32", seed=2)
    prob = cp.Problem(1, H, 1, n, 64, seg, seg, 1, torch.float32)
    ws = cp.alloc_workspace(prob)
    Qd, Kd, Vd = Q.cuda(), K.cuda(), V.cuda()
    idx = torch.zeros((1, H, 1, 1), dtype=torch.int32, device="cuda")
    cnt = torch.ones((1, H, 1), dtype=torch.int32, device="cuda")
    O = cp.attention(prob, Qd, Kd, Vd, idx, cnt, ws)
    Od = cp.dense_attention(prob, Qd, Kd, Vd, ws)
    assert cp.device_status(ws) == 0
    O_ref, _ = oracle.dense_attention(Q, K, V, f32(0.125))
    assert_close(O, O_ref, V, "f32")
    assert_close(Od, O_ref, V, "f32")


def test_value_that_is_not_finite_reaches_only_the_rows_that_see_it():
    n, seg, blk, k = 700, 256, 32, 12
    Q, K, V = make_uniform_qkv(1, 2, 1, n, 64, dtype="f32", seed=1)
    prob = cp.Problem(1, 2, 1, n, 64, seg, blk, k, torch.float32)
    ws = cp.alloc_workspace(prob)
    Vf = V.clone()
    V[0, 0, 300, 5] = float("inf")
    Vf[0, 0, 300, 5] = 0
    O = cp.dense_attention(prob, Q.cuda(), K.cuda(), V.cuda(), ws).cpu().numpy()
    assert cp.device_status(ws) == 0
    assert np.isfinite(O[:, :, :300]).all() and not np.isfinite(O[:, :, 300:, 5]).any()
    O_ref, _ = oracle.dense_attention(Q, K, Vf, f32(0.125))
    assert_close(torch.from_numpy(O[:, :, :300]), O_ref[:, :, :300], Vf, "f32")
