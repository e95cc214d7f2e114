"""Block criticality of the newest token against the fp64 oracle: block sizes a warp takes and larger ones, ragged lengths, every
type and head size, group sizes on both sides of the workspace rule, strided keys, and the longest rows of blocks."""
import numpy as np
import pytest
import torch

import oracle
from paper_2409_12490_b200 import binding as cp
from paper_2409_12490_b200.inputs import make_uniform_qkv

from helpers import f32

pytestmark = pytest.mark.gpu

TDT = {"bf16": torch.bfloat16, "f16": torch.float16, "f32": torch.float32}


@pytest.mark.parametrize("dtype,d", [("bf16", 128), ("f16", 128), ("bf16", 64), ("f16", 64), ("f32", 64), ("f32", 128)])
@pytest.mark.parametrize("B,Hkv,g,n,blk,k", [
    (1, 1, 1, 1, 32, 4), (2, 2, 4, 257, 32, 5), (1, 2, 3, 1000, 16, 9), (1, 1, 40, 700, 64, 3), (3, 1, 8, 2049, 128, 20),
    (1, 1, 2, 4096, 256, 6), (1, 1, 1, 4100, 4, 64), (1, 1, 2, 4096, 1, 64)])
def test_scores_and_list_match_the_oracle(dtype, d, B, Hkv, g, n, blk, k):
    Hq = Hkv * g
    Q, K, V = make_uniform_qkv(B, Hq, Hkv, n, d, dtype=dtype, seed=n + g)
    prob = cp.Problem(B, Hq, Hkv, n, d, blk, blk, k, TDT[dtype])
    ws = cp.alloc_workspace(prob)
    q = Q[:, :, -1].contiguous()
    Kd = K.permute(0, 2, 1, 3).contiguous().cuda().permute(0, 2, 1, 3)         # [batch, tokens, heads, d] storage
    S = cp.decode_estimate(prob, q.cuda(), Kd, ws)
    idx, cnt = cp.decode_select(prob, S, ws)
    assert cp.device_status(ws) == 0
    S_ref = oracle.decode_estimate(q, K, blk, est_scale=f32(1.0))
    assert np.abs(S.cpu().numpy() - S_ref).max() <= 1e-9
    idx_ref, cnt_ref = oracle.decode_select(S.cpu().numpy(), k)
    assert np.array_equal(idx.cpu().numpy(), idx_ref) and np.array_equal(cnt.cpu().numpy(), cnt_ref)


@pytest.mark.parametrize("g", [96, 97, 128, 129])
def test_large_query_groups_in_fp32(g):
    """Up to 128 fp32 heads of 128 channels per KV head share the pass over the key cache (their queries fill up to 64 KB of shared
    memory, 48 KB at 96 heads); one head more takes the general kernels."""
    n, blk, k = 700, 64, 3
    Q, K, V = make_uniform_qkv(1, g, 1, n, 128, dtype="f32", seed=g)
    prob = cp.Problem(1, g, 1, n, 128, blk, blk, k, torch.float32)
    ws = cp.alloc_workspace(prob)
    q = Q[:, :, -1].contiguous()
    S = cp.decode_estimate(prob, q.cuda(), K.cuda(), ws)
    assert cp.device_status(ws) == 0
    assert np.abs(S.cpu().numpy() - oracle.decode_estimate(q, K, blk, est_scale=f32(1.0))).max() <= 1e-9


def _bad_values(what, q, K, blk):
    inf, nan = float("inf"), float("nan")
    if what == "channel of a block NaN":
        K[0, 0, 3 * blk:4 * blk, 7] = nan
    elif what == "one key +inf":
        K[0, 0, 3 * blk + blk // 2, 7] = inf
    elif what == "one key -inf":
        K[0, 0, 3 * blk + blk // 2, 7] = -inf
    elif what == "NaN logits of one block":          # infinities of both signs in the representatives of two channels
        K[0, 0, 3 * blk, 7] = K[0, 0, 3 * blk + 1, 9] = inf
        K[0, 0, 3 * blk, 9] = K[0, 0, 3 * blk + 1, 7] = -inf
        q[0, 0, 7], q[0, 0, 9] = 1.0, -1.0
        q[0, 1, 7], q[0, 1, 9] = 1.0, 1.0
    elif what == "q inf":
        q[0, 1, 3] = inf
    elif what == "keys NaN":
        K[...] = nan
    return q, K


@pytest.mark.parametrize("dtype,d", [("f32", 64), ("bf16", 64), ("f32", 128)])
@pytest.mark.parametrize("blk,g", [(2, 2), (32, 4), (128, 2)])
@pytest.mark.parametrize("what", ["channel of a block NaN", "one key +inf", "one key -inf", "NaN logits of one block", "q inf", "keys NaN"])
def test_values_that_are_not_finite_follow_the_general_kernel(dtype, d, blk, g, what):
    """The last segment of a prefill may hold the newest token alone: its row of the general score kernel is then the decoding row,
    and what NaN and infinite logits do to the other blocks has to be the same."""
    n = 20 * blk + 1
    Q, K, V = make_uniform_qkv(1, g, 1, n, d, dtype=dtype, seed=blk)
    q = Q[:, :, -1].clone()
    q, K = _bad_values(what, q, K.clone(), blk)
    Q[:, :, -1] = q
    prob = cp.Problem(1, g, 1, n, d, blk, blk, 4, TDT[dtype])
    ws = cp.alloc_workspace(prob)
    row = cp.estimate(prob, Q.cuda(), K.cuda(), ws)[:, :, -1].cpu().numpy()
    S = cp.decode_estimate(prob, q.contiguous().cuda(), K.cuda(), ws).cpu().numpy()
    assert cp.device_status(ws) == 0
    for kind in (np.isnan, np.isposinf, np.isneginf):
        assert np.array_equal(kind(S), kind(row)), kind.__name__
    fin = np.isfinite(row)
    assert np.abs(S[fin] - row[fin]).max(initial=0.0) <= 1e-9


@pytest.mark.parametrize("B,Hkv,g,n,blk", [
    (1, 2, 4, 256 * 16, 16), (1, 2, 4, 256 * 16 + 1, 16),    # 2 g n2 = 2048 and one block more
    (1, 56, 1, 300, 32), (3, 19, 1, 300, 32),                 # 56 KV heads have a counter behind the status word each; 57 do not
    (1, 1, 32, 1024, 32), (1, 1, 33, 500, 32)])
def test_rows_normalised_behind_their_logits_or_by_a_kernel_of_their_own(B, Hkv, g, n, blk):
    """Two calls on one workspace (the counters start from zero again), another problem between them."""
    Q, K, V = make_uniform_qkv(B, Hkv * g, Hkv, n, 64, dtype="bf16", seed=n + g)
    prob = cp.Problem(B, Hkv * g, Hkv, n, 64, blk, blk, 2, torch.bfloat16)
    ws = cp.alloc_workspace(prob)
    q, Kd = Q[:, :, -1].contiguous(), K.cuda()
    S_ref = oracle.decode_estimate(q, K, blk, est_scale=f32(1.0))
    small = cp.Problem(1, g, 1, 100, 64, blk, blk, 2, torch.bfloat16)
    for _ in range(2):
        S = cp.decode_estimate(prob, q.cuda(), Kd, ws)
        cp.decode_estimate(small, q[:1, :g].contiguous().cuda(), Kd[:1, :1, :100].contiguous(), ws)
        assert cp.device_status(ws) == 0
        assert np.abs(S.cpu().numpy() - S_ref).max() <= 1e-9


@pytest.mark.parametrize("Hkv,g,n,blk", [(8, 4, 256 * 8, 8), (2, 4, 300, 32), (1, 1, 5, 32)])
def test_decoding_needs_nothing_of_what_the_workspace_holds(Hkv, g, n, blk):
    Q, K, V = make_uniform_qkv(1, Hkv * g, Hkv, n, 128, dtype="bf16", seed=n)
    prob = cp.Problem(1, Hkv * g, Hkv, n, 128, blk, blk, 2, torch.bfloat16)
    q, Kd = Q[:, :, -1].contiguous().cuda(), K.cuda()
    ws = cp.alloc_workspace(prob)
    S = cp.decode_estimate(prob, q, Kd, ws)
    assert torch.equal(S, cp.decode_estimate(prob, q, Kd, torch.full_like(ws, 1)))


@pytest.mark.parametrize("dtype,d", [("bf16", 128), ("f16", 64), ("f32", 128), ("f32", 64)])
@pytest.mark.parametrize("B,Hkv,g,n2,blk", [
    (1, 1, 1, 8, 4), (1, 2, 3, 9, 4), (2, 1, 4, 64, 4), (1, 2, 5, 65, 4), (1, 1, 8, 255, 4), (2, 3, 7, 256, 4),    # 1 to 16 CTAs of 8 to 16 warps
    (1, 1, 9, 256, 4), (1, 2, 4, 257, 4), (2, 65, 1, 130, 4),                                                     # a head, a block, a batch too many
    (1, 13, 2, 250, 32), (2, 75, 1, 40, 32)])                                                                     # two blocks per warp where these are long
def test_short_rows_over_clusters_of_every_size(dtype, d, B, Hkv, g, n2, blk):
    """The last block has one row."""
    n = (n2 - 1) * blk + 1
    Q, K, V = make_uniform_qkv(B, Hkv * g, Hkv, n, d, dtype=dtype, seed=n2 + g)
    prob = cp.Problem(B, Hkv * g, Hkv, n, d, blk, blk, 2, TDT[dtype])
    ws = cp.alloc_workspace(prob)
    q = Q[:, :, -1].contiguous()
    S = cp.decode_estimate(prob, q.cuda(), K.cuda(), ws)
    assert np.abs(S.cpu().numpy() - oracle.decode_estimate(q, K, blk, est_scale=f32(1.0))).max() <= 1e-9


@pytest.mark.parametrize("n", [300, 8000, 8200])
def test_decoding_replays_from_a_cuda_graph(n):
    """One launch of clusters of 2 or 16 CTAs, and two kernels, captured and replayed over other keys."""
    prob = cp.Problem(1, 8, 2, n, 128, 32, 32, 8, torch.bfloat16)
    (Q, K, _), (Q1, K1, _) = (make_uniform_qkv(1, 8, 2, n, 128, dtype="bf16", seed=x) for x in (1, 2))
    q, Kd, ws = Q[:, :, -1].contiguous().cuda(), K.cuda(), cp.alloc_workspace(prob)
    cp.decode_estimate(prob, q, Kd, ws)
    S = torch.empty(1, 8, prob.n2, dtype=torch.float64, device="cuda")
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        cp.decode_estimate(prob, q, Kd, ws, S_out=S)
    q.copy_(Q1[:, :, -1]); Kd.copy_(K1)
    graph.replay()
    assert torch.equal(S, cp.decode_estimate(prob, q, Kd, ws))
