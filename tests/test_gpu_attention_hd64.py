"""The tensor-core attention kernel on heads of 64 channels (probabilities held as sums of two or three 16-bit values) against
the fp64 oracle: tile edges, ragged tails, odd tile counts, one-unit and long problems, and values that are not finite."""
import numpy as np
import pytest
import torch

import oracle
from paper_2409_12490_b200 import CONFIGS, binding as cp
from paper_2409_12490_b200.inputs import make_qkv, make_uniform_qkv

from helpers import f32

pytestmark = pytest.mark.gpu

SM = f32(1.0 / np.sqrt(64))
TDT = {"bf16": torch.bfloat16, "f16": torch.float16}


def layer(dtype, B, Hq, Hkv, n, seg, blk, k, seed=3):
    Q, K, V = make_uniform_qkv(B, Hq, Hkv, n, 64, dtype=dtype, seed=seed)
    prob = cp.Problem(B, Hq, Hkv, n, 64, seg, blk, k, TDT[dtype])
    ws = cp.alloc_workspace(prob)
    Qd, Kd, Vd = Q.cuda(), K.cuda(), V.cuda()
    idx, cnt = cp.select(prob, cp.estimate(prob, Qd, Kd, ws), ws)
    return Q, K, V, prob, ws, Qd, Kd, Vd, idx, cnt


def assert_close(O, O_ref, V, dtype):
    """|O_gpu - O| <= u |O| + e max|V|: u is the unit roundoff of the one rounding of O; e covers the split of P (2^-24 for
    bf16, 2^-22 for fp16), exponentials and logits in fp32 (2^-20 each) and fp32 accumulation over up to 2^11 keys (2^-16 at
    most).  A single 16-bit rounding of P (2^-9 max|V| and 2^-12 max|V|) would not pass on averages of this length."""
    u, e = {"bf16": (2.0 ** -8, 2.0 ** -15), "f16": (2.0 ** -11, 2.0 ** -15)}[dtype]
    err = np.abs(O.float().cpu().numpy().astype(np.float64) - O_ref)
    assert (err <= u * np.abs(O_ref) + e * float(V.float().abs().max())).all(), float(err.max())


@pytest.mark.parametrize("dtype", ["bf16", "f16"])
@pytest.mark.parametrize("B,Hq,Hkv,n,seg,blk,k", [
    (1, 2, 1, 1, 128, 32, 4), (1, 4, 2, 127, 128, 32, 5), (2, 2, 2, 129, 128, 64, 3), (1, 4, 1, 640, 384, 128, 4),
    (1, 2, 1, 1301, 512, 32, 19), (3, 4, 2, 2048, 256, 64, 9), (1, 2, 2, 4099, 1024, 128, 17)])
def test_sparse_and_dense_match_the_oracle(dtype, B, Hq, Hkv, n, seg, blk, k):
    Q, K, V, prob, ws, Qd, Kd, Vd, idx, cnt = layer(dtype, B, Hq, Hkv, n, seg, blk, k)
    O, lse = cp.attention(prob, Qd, Kd, Vd, idx, cnt, ws, want_lse=True)
    Od = cp.dense_attention(prob, Qd, Kd, Vd, ws)
    assert cp.device_status(ws) == 0
    O_ref, lse_ref = oracle.sparse_attention(Q, K, V, idx.cpu().numpy(), cnt.cpu().numpy(), seg, blk, SM)
    assert_close(O, O_ref, V, dtype)
    assert np.abs(lse.cpu().numpy() - lse_ref).max() <= 1e-4
    assert_close(Od, oracle.dense_attention(Q, K, V, SM)[0], V, dtype)


@pytest.mark.parametrize("positive", [False, True])
@pytest.mark.parametrize("dtype,share", [("bf16", 2.0 ** -11), ("f16", 2.0 ** -8)])
def test_outputs_are_those_of_32_bit_arithmetic(dtype, share, positive):
    """Before its rounding to 16 bits (spacing 2^-8 to 2^-7 of the output in bf16, 2^-11 to 2^-10 in fp16) O is good to 2^-19 of its
    size: roundings in fp32 over 8000 keys, not a chain of accumulations towards zero (2^-16 when the values have one sign).  So
    at most 2^-19 / 2^-8 or 2^-19 / 2^-11 of the outputs are rounded otherwise than the fp64 result."""
    n = 8000
    cfg = CONFIGS["C2"].with_(name="hd64", seq_len=n, n_q_heads=4, n_kv_heads=2, head_dim=64, segment_size=512, block_size=64,
                              budget_tokens=1024, n_clusters=16, dtype=dtype)
    Q, K, V = (t.cuda() for t in make_qkv(cfg))
    V = V.abs() if positive else V
    prob = cp.Problem.from_config(cfg)
    ws = cp.alloc_workspace(prob)
    O = cp.dense_attention(prob, Q, K, V, ws)
    assert cp.device_status(ws) == 0
    future = torch.ones((n, n), dtype=torch.bool, device="cuda").triu(1)
    off = 0.0
    for h in range(4):
        s = ((Q[0, h].double() @ K[0, h // 2].double().T) * SM).masked_fill_(future, -float("inf"))
        off += float((O[0, h] != (torch.softmax(s, 1) @ V[0, h // 2].double()).to(O.dtype)).double().mean()) / 4
    assert off <= share, off


def launched_grids(call):
    """gridDim.x of every kernel that `call` enqueues, from a captured graph (nothing runs)."""
    from cuda.bindings import driver as cu
    g = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(g):
        keep = call()
    raw = cu.CUgraph(g.raw_cuda_graph())
    n = cu.cuGraphGetNodes(raw, 0)[2]
    grids = []
    for node in cu.cuGraphGetNodes(raw, n)[1][:n]:
        if cu.cuGraphNodeGetType(node)[1] == cu.CUgraphNodeType.CU_GRAPH_NODE_TYPE_KERNEL:
            rc, params = cu.cuGraphKernelNodeGetParams(node)
            assert rc == cu.CUresult.CUDA_SUCCESS, rc
            grids.append(params.gridDimX)
    del keep
    return grids


@pytest.mark.parametrize("B,n", [(1, 1), (2, 300), (1, 1301)])
def test_segment_far_longer_than_the_sequence(B, n):
    """Units are counted over the rows there are, not over the segment's 2^20."""
    seg, blk = 1 << 20, 128
    Q, K, V, prob, ws, Qd, Kd, Vd, idx, cnt = layer("f16", B, 4, 2, n, seg, blk, seg // blk)
    O = cp.attention(prob, Qd, Kd, Vd, idx, cnt, ws)
    assert cp.device_status(ws) == 0
    assert_close(O, oracle.dense_attention(Q, K, V, SM)[0], V, "f16")
    assert launched_grids(lambda: cp.attention(prob, Qd, Kd, Vd, idx, cnt, ws)) == [B * 4 * -(-n // 256)]


@pytest.mark.parametrize("dtype", ["bf16", "f16"])
def test_value_that_is_not_finite_reaches_only_the_rows_that_see_it(dtype):
    n, seg, blk, k = 700, 256, 32, 12
    Q, K, V, prob, ws, Qd, Kd, Vd, idx, cnt = layer(dtype, 1, 2, 1, n, seg, blk, k)
    bad = 300
    Vd[0, 0, bad, 5] = float("inf")
    Vf = V.clone()
    Vf[0, 0, bad, 5] = 0
    for dense in (False, True):
        O = cp.dense_attention(prob, Qd, Kd, Vd, ws) if dense else cp.attention(prob, Qd, Kd, Vd, idx, cnt, ws)
        assert cp.device_status(ws) == 0
        O = O.float().cpu().numpy()
        li = idx.cpu().numpy()
        sees = np.zeros((2, n), dtype=bool)
        for h in range(2):
            for t in range(bad, n):
                sees[h, t] = dense or bad // blk in li[0, h, t // seg]
        assert np.isfinite(O[0][~sees]).all() and not np.isfinite(O[0][sees][:, 5]).any()
        O_ref = oracle.dense_attention(Q, K, Vf, SM)[0] if dense else oracle.sparse_attention(Q, K, Vf, li, cnt.cpu().numpy(), seg, blk, SM)[0]
        assert_close(torch.from_numpy(O[0][~sees]), O_ref[0][~sees], V, dtype)


@pytest.mark.parametrize("dtype", ["bf16", "f16"])
@pytest.mark.parametrize("storage", ["heads share their keys", "batches share their keys", "queries shared", "tokens first"])
def test_strides(dtype, storage):
    """Strides of 0 (expanded tensors), a token stride that is larger than the head stride, and the stride of a dimension of extent 1,
    which nothing reads, at 2^40 bytes."""
    B, H, n, seg, blk, k = 2, 3, 700, 256, 64, 6
    Q, K, V = make_uniform_qkv(B, H, H, n, 64, dtype=dtype, seed=5)
    if storage == "heads share their keys":
        K, V = K[:, :1].expand(-1, H, -1, -1), V[:, :1].expand(-1, H, -1, -1)
    elif storage == "batches share their keys":
        K, V = K[:1].expand(B, -1, -1, -1), V[:1].expand(B, -1, -1, -1)
    elif storage == "queries shared":
        Q = Q[:, :1].expand(-1, H, -1, -1)
    dense = [t.contiguous().cuda() for t in (Q, K, V)]
    if storage == "tokens first":
        Qd, Kd, Vd = (t.permute(0, 2, 1, 3).contiguous().permute(0, 2, 1, 3) for t in dense)
        Qd, Kd, Vd = (t[:1].as_strided((1, H, n, 64), (1 << 39, 64, H * 64, 1)) for t in (Qd, Kd, Vd))
        dense = [t[:1] for t in dense]
    else:
        Qd, Kd, Vd = (t.cuda() if t.is_contiguous() else _expand_like(t) for t in (Q, K, V))
    prob = cp.Problem(Qd.shape[0], H, H, n, 64, seg, blk, k, TDT[dtype])
    ws = cp.alloc_workspace(prob)
    idx, cnt = cp.select(prob, cp.estimate(prob, dense[0], dense[1], ws), ws)
    O = torch.empty_like(dense[0])
    for a, b in ((cp.attention(prob, Qd, Kd, Vd, idx, cnt, ws, O=O.clone()), cp.attention(prob, *dense, idx, cnt, ws)),
                 (cp.dense_attention(prob, Qd, Kd, Vd, ws, O=O.clone()), cp.dense_attention(prob, *dense, ws))):
        assert torch.equal(a, b)
    assert cp.device_status(ws) == 0


def _expand_like(t):
    """The expanded CPU tensor's one copy on the device, expanded again."""
    return t[tuple(slice(0, 1) if s == 0 else slice(None) for s in t.stride())].contiguous().cuda().expand(t.shape)


def test_value_that_is_not_finite_at_the_end_of_a_long_sequence():
    """The last 300 rows of 1.3 M tokens see an infinite value and are evaluated one by one, over more keys than the kernel's waits
    would sit out for a thread per row: the call ends without an error, every row before them is finite, and the rows are those of
    the formula."""
    n, bad = 1_300_000, 1_300_000 - 300
    gen = torch.Generator(device="cuda").manual_seed(4)
    Q, K, V = (torch.randn((1, 1, n, 64), generator=gen, device="cuda").to(torch.bfloat16) for _ in range(3))
    V[0, 0, bad, 5] = float("inf")
    prob = cp.Problem(1, 1, 1, n, 64, 1024, 128, 16, torch.bfloat16)
    ws = cp.alloc_workspace(prob)
    O, lse = cp.dense_attention(prob, Q, K, V, ws, want_lse=True)
    assert cp.device_status(ws) == 0
    assert torch.isfinite(O[0, 0, :bad]).all() and torch.isposinf(O[0, 0, bad:, 5]).all()
    keep = torch.arange(64, device="cuda") != 5
    assert torch.isfinite(O[0, 0, bad:][:, keep]).all()
    for t in (bad - 1, bad, n - 1):
        s = (K[0, 0, :t + 1].double() @ Q[0, 0, t].double()) * SM
        ref = torch.softmax(s, 0) @ V[0, 0, :t + 1].double()
        assert abs(float(torch.logsumexp(s, 0)) - float(lse[0, 0, t])) <= 1e-4
        # outputs of about 1e-3: one rounding to bf16, and fp32 sums over 2^20 keys that add up to 1 (2^-17 of max|V| ~ 5)
        assert (O[0, 0, t].double() - ref)[keep].abs().max() <= 2.0 ** -8 * ref[keep].abs().max() + 2.0 ** -17 * 5
