"""More sequences than one launch takes, workspaces that hold them in several groups, both head sizes, sequences on either score
path: every sequence equals its single-sequence call bit for bit, and a neighbour's values that are not finite do not reach it."""
import numpy as np
import pytest
import torch

from paper_2409_12490_b200 import binding as cp
from paper_2409_12490_b200.inputs import make_uniform_qkv

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,dtype", [(128, torch.bfloat16), (64, torch.float16)])
@pytest.mark.parametrize("lens", [[1], [1, 128, 129], [17 + 61 * i for i in range(19)], [1500, 33, 2049, 256] * 9,
                                  [66000, 67000, 140000]])      # more segments than one launch's table of units
def test_each_sequence_equals_its_own_call(d, dtype, lens):
    Hq, Hkv, seg, blk, k = (4, 2, 256, 32, 12) if max(lens) < 5000 else (1, 1, 128, 128, 3)
    total = sum(lens)
    Q, K, V = make_uniform_qkv(1, Hq, Hkv, total, d, dtype={torch.bfloat16: "bf16", torch.float16: "f16"}[dtype], seed=len(lens))
    pack = lambda t: t[0].permute(1, 0, 2).contiguous().cuda().permute(1, 0, 2)
    Q, K, V = pack(Q), pack(K), pack(V)
    cu = [0] + np.cumsum(lens).tolist()
    if len(lens) > 1:
        V[:, cu[1]:cu[2]] = float("inf")                       # the second sequence's values
    prob = cp.Problem(1, Hq, Hkv, max(lens), d, seg, blk, k, dtype)
    ws = cp.alloc_workspace(prob)
    O, S, idx, cnt, _, lse = cp.prefill_varlen(prob, cu, Q, K, V, ws, want_lse=True)
    assert cp.device_status(ws) == 0
    for i, (lo, hi) in enumerate(zip(cu[:-1], cu[1:])):
        one = cp.Problem(1, Hq, Hkv, hi - lo, d, seg, blk, k, dtype)
        part = [t[None, :, lo:hi] for t in (Q, K, V)]
        S1 = cp.estimate(one, part[0], part[1], ws)
        idx1, cnt1 = cp.select(one, S1, ws)
        O1, lse1 = cp.attention(one, *part, idx1, cnt1, ws, want_lse=True)
        assert torch.equal(S[i], S1[0]) and torch.equal(idx[i], idx1[0]) and torch.equal(cnt[i], cnt1[0])
        assert torch.equal(lse[Hq * lo:Hq * hi].view(Hq, hi - lo), lse1[0])
        if i == 1:
            assert not torch.isfinite(O[:, lo:hi].float()).any()
        else:
            assert torch.equal(O[:, lo:hi], O1[0]) and torch.isfinite(O[:, lo:hi].float()).all()


@pytest.mark.parametrize("flags,dtype,d", [(cp.FLAG_FORCE_SPLIT_SCORE, torch.bfloat16, 128), (0, torch.float32, 64),
                                           (cp.FLAG_SHARED_GROUP_LISTS | cp.FLAG_MASK_BEFORE_SOFTMAX, torch.float16, 128)])
@pytest.mark.parametrize("room", [1, 20])                      # workspaces of the longest sequence
def test_fused_layers_equal_their_own_calls(flags, dtype, d, room):
    lens, Hq, Hkv, seg, blk, k = [1500, 33, 2049, 256, 700] * 4, 4, 2, 256, 4, 80
    name = {torch.bfloat16: "bf16", torch.float16: "f16", torch.float32: "f32"}[dtype]
    total, cu = sum(lens), [0] + np.cumsum(lens).tolist()
    layers = [[t[0].cuda() for t in make_uniform_qkv(1, Hq, Hkv, total, d, dtype=name, seed=s)] for s in (1, 2)]
    prob = cp.Problem(1, Hq, Hkv, max(lens), d, seg, blk, k, dtype, flags=flags)
    ws = torch.zeros(room * cp.workspace_bytes(prob), dtype=torch.uint8, device="cuda")
    first = cp.prefill_varlen(prob, cu, *layers[0], ws)
    O, S, idx, cnt, _ = cp.prefill_varlen(prob, cu, *layers[1], ws, S_prev=first[4])
    assert cp.device_status(ws) == 0
    for i, (lo, hi) in enumerate(zip(cu[:-1], cu[1:])):
        one = cp.Problem(1, Hq, Hkv, hi - lo, d, seg, blk, k, dtype, flags=flags)
        O1, S1, idx1, cnt1 = cp.prefill_layer(one, *[t[None, :, lo:hi] for t in layers[1]], ws, S_prev=first[1][i][None])
        assert torch.equal(S[i], S1[0]) and torch.equal(idx[i], idx1[0]) and torch.equal(cnt[i], cnt1[0])
        assert torch.equal(O[:, lo:hi], O1[0])


def test_batch_whose_scores_need_clusters_of_every_size():
    """Four heads per CTA, blocks of 4 tokens: up to 1064 blocks fit one CTA's shared memory, 2128 two, 4256 four, 8192 eight; half of that are
    split twice as often where that makes no more than 148 CTAs.  Two sequences or more of each size (1: 33, 1500; 2: 3000, 4265, 4300; 4: 8000,
    5000, 9000, 17000; 8: 18000, 20000) in one batch, so that every cluster launch holds several sequences with offsets of their own."""
    lens, Hq, Hkv, d, seg, blk, k = [3000, 8000, 18000, 5000, 33, 9000, 4265, 20000, 4300, 1500, 17000], 4, 1, 64, 256, 4, 64
    total, cu = sum(lens), [0] + np.cumsum(lens).tolist()
    layers = [[t[0].cuda() for t in make_uniform_qkv(1, Hq, Hkv, total, d, dtype="f32", seed=s)] for s in (3, 4)]
    prob = cp.Problem(1, Hq, Hkv, max(lens), d, seg, blk, k, torch.float32)
    ws = torch.zeros(8 * cp.workspace_bytes(prob), dtype=torch.uint8, device="cuda")
    first = cp.prefill_varlen(prob, cu, *layers[0], ws)
    O, S, idx, cnt, _ = cp.prefill_varlen(prob, cu, *layers[1], ws, S_prev=first[4])
    assert cp.device_status(ws) == 0
    for i, (lo, hi) in enumerate(zip(cu[:-1], cu[1:])):
        one = cp.Problem(1, Hq, Hkv, hi - lo, d, seg, blk, k, torch.float32)
        S0 = cp.estimate(one, layers[0][0][None, :, lo:hi], layers[0][1][None, :, lo:hi], ws)
        O1, S1, idx1, cnt1 = cp.prefill_layer(one, *[t[None, :, lo:hi] for t in layers[1]], ws, S_prev=S0)
        assert torch.equal(first[1][i], S0[0]) and torch.equal(S[i], S1[0])
        assert torch.equal(idx[i], idx1[0]) and torch.equal(cnt[i], cnt1[0]) and torch.equal(O[:, lo:hi], O1[0])
