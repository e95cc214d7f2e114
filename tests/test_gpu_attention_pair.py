"""The attention kernel of CTA pairs (launches of few or of short units) against the fp64 oracle at the edges of its tiles, and against the
single-CTA kernel, whose results it has to give bit for bit."""
import numpy as np
import pytest
import torch

import oracle
from paper_2409_12490_b200 import binding as cp
from paper_2409_12490_b200.inputs import make_uniform_qkv

from helpers import f32

pytestmark = pytest.mark.gpu

SM = f32(1.0 / np.sqrt(128))
TDT = {"bf16": torch.bfloat16, "f16": torch.float16}


def assert_close(O, O_ref, V, dtype):
    """|O_gpu - O| <= u (|O| + max|V|) + 2^-13 max|V|: one rounding of O and one of every probability to 16 bits (unit roundoff u), the
    polynomial exponentials (7.5e-5), and 2^-15 for logits, exponentials and sums in fp32."""
    u = {"bf16": 2.0 ** -9, "f16": 2.0 ** -12}[dtype] * (1 + 2.0 ** -7)
    vmax = float(V.float().abs().max())
    err = np.abs(O.float().cpu().numpy().astype(np.float64) - O_ref)
    assert (err <= u * (np.abs(O_ref) + vmax) + 2.0 ** -13 * vmax).all(), float(err.max())


@pytest.mark.parametrize("dtype", ["bf16", "f16"])
@pytest.mark.parametrize("B,Hq,Hkv,n,seg,blk,k", [
    (1, 1, 1, 1, 256, 32, 8), (1, 2, 1, 127, 256, 64, 5), (2, 2, 2, 129, 256, 128, 2), (1, 4, 2, 257, 256, 32, 9),
    (3, 4, 1, 640, 512, 64, 9), (1, 8, 2, 1300, 512, 32, 32), (1, 4, 4, 2049, 256, 128, 16), (1, 2, 1, 4096, 1024, 32, 77)])
def test_sparse_and_dense_match_the_oracle(dtype, B, Hq, Hkv, n, seg, blk, k):
    Q, K, V = make_uniform_qkv(B, Hq, Hkv, n, 128, dtype=dtype, seed=n)
    prob = cp.Problem(B, Hq, Hkv, n, 128, seg, blk, k, TDT[dtype])
    ws = cp.alloc_workspace(prob)
    Qd, Kd, Vd = Q.cuda(), K.cuda(), V.cuda()
    idx, cnt = cp.select(prob, cp.estimate(prob, Qd, Kd, ws), ws)
    O, lse = cp.attention(prob, Qd, Kd, Vd, idx, cnt, ws, want_lse=True)
    Od = cp.dense_attention(prob, Qd, Kd, Vd, ws)
    assert cp.device_status(ws) == 0
    O_ref, lse_ref = oracle.sparse_attention(Q, K, V, idx.cpu().numpy(), cnt.cpu().numpy(), seg, blk, SM)
    assert_close(O, O_ref, V, dtype)
    assert np.abs(lse.cpu().numpy() - lse_ref).max() <= 1e-4
    assert_close(Od, oracle.dense_attention(Q, K, V, SM)[0], V, dtype)


@pytest.mark.parametrize("dtype", ["bf16", "f16"])
@pytest.mark.parametrize("B,n,seg,blk,k", [(9, 2049, 256, 64, 32), (9, 3000, 512, 128, 16), (9, 2561, 1024, 32, 50), (30, 2049, 256, 32, 32)])
def test_few_and_many_units_give_the_same_bits(dtype, B, n, seg, blk, k):
    """One item of the batch alone (few units: pairs of CTAs) and all of them (more than 444 units, short ones more than 2072: one CTA each).
    Logits of up to some 30 make the reference maximum move."""
    Hq, Hkv = 8, 2
    Q, K, V = (t.cuda() for t in make_uniform_qkv(B, Hq, Hkv, n, 128, dtype=dtype, seed=n))
    Q = Q * 3
    K = K * torch.linspace(0.2, 3.0, n, device="cuda").to(K.dtype).view(1, 1, n, 1)
    out = {}
    for name, b in (("all", slice(0, B)), ("one", slice(4, 5))):
        q, kk, v = Q[b].contiguous(), K[b].contiguous(), V[b].contiguous()
        prob = cp.Problem(q.shape[0], Hq, Hkv, n, 128, seg, blk, k, TDT[dtype])
        ws = cp.alloc_workspace(prob)
        idx, cnt = cp.select(prob, cp.estimate(prob, q, kk, ws), ws)
        out[name] = cp.attention(prob, q, kk, v, idx, cnt, ws, want_lse=True) + cp.dense_attention(prob, q, kk, v, ws, want_lse=True)
        assert cp.device_status(ws) == 0
    for a, b in zip(out["all"], out["one"]):
        assert torch.equal(a[4], b[0])


def test_keys_that_only_the_second_tile_sees_stay_out_of_the_first():
    """A unit's last tile of keys lies after its first 128 rows; an infinite value there must not reach them as 0 x inf."""
    n = 512
    Q, K, V = (t.cuda() for t in make_uniform_qkv(1, 2, 1, n, 128, seed=5))
    prob = cp.Problem(1, 2, 1, n, 128, 256, 64, 6, torch.bfloat16)
    ws = cp.alloc_workspace(prob)
    idx, cnt = cp.select(prob, cp.estimate(prob, Q, K, ws), ws)
    W = V.clone()
    W[:, :, 400] = float("inf")                       # in the last tile of the unit of rows 256 to 511
    for f in (lambda v: cp.attention(prob, Q, K, v, idx, cnt, ws), lambda v: cp.dense_attention(prob, Q, K, v, ws)):
        clean, odd = f(V), f(W)
        assert torch.equal(clean[:, :, :384], odd[:, :, :384]) and not torch.isfinite(odd[:, :, 400:]).any()
    assert cp.device_status(ws) == 0


def mixed_lists(Hq, n, seg, blk, k, seed, broken):
    """Lists of length 0, 1 and k in every order, any visible blocks among them; broken: some that break their contract."""
    rng = np.random.default_rng(seed)
    n1, n2, r = -(-n // seg), -(-n // blk), seg // blk
    idx = np.full((1, Hq, n1, k), -1, dtype=np.int32)
    cnt = np.zeros((1, Hq, n1), dtype=np.int32)
    for h in range(Hq):
        for j in range(n1):
            own = list(range(j * r, min(n2, (j + 1) * r)))
            mode = rng.choice(["empty", "empty", "one", "standard", "standard", "any", "broken"])
            if mode == "empty":
                sel = []
            elif mode == "one":
                sel = [int(rng.integers(own[-1] + 1))]
            elif mode == "any":
                sel = sorted(rng.choice(own[-1] + 1, size=min(k, own[-1] + 1), replace=False).tolist())
            else:
                sel = sorted(rng.choice(j * r, size=min(k - r, j * r), replace=False).tolist() if j else []) + own
                if mode == "broken" and broken:
                    sel[-1] = n2 + 1000
            cnt[0, h, j] = len(sel)
            idx[0, h, j, :len(sel)] = sel
    return torch.from_numpy(idx), torch.from_numpy(cnt)


@pytest.mark.parametrize("broken", [False, True])
@pytest.mark.parametrize("dtype,blk,k,items,Hq,Hkv,n", [("bf16", 32, 32, 7, 16, 4, 5000), ("f16", 128, 8, 7, 16, 4, 5000), ("bf16", 64, 32, 3, 2, 1, 27000)])
def test_mixed_lists_over_many_units(dtype, blk, k, items, Hq, Hkv, n, broken):
    """Each pair of CTAs draws three units or more, with empty and one-block lists before and behind full ones.  One item alone (320 short
    or 212 long units: pairs) and in a batch (2240 short units, 636 long ones: one CTA each); rows of a broken list are left as they were by both."""
    seg = 256
    Q, K, V = (t.cuda() for t in make_uniform_qkv(items, Hq, Hkv, n, 128, dtype=dtype, seed=k))
    lists = [mixed_lists(Hq, n, seg, blk, k, 10 * i + k, broken) for i in range(items)]
    idx, cnt = (torch.cat([x[i] for x in lists]).cuda() for i in (0, 1))

    def run(b):
        q, kk, v = Q[b].contiguous(), K[b].contiguous(), V[b].contiguous()
        prob = cp.Problem(q.shape[0], Hq, Hkv, n, 128, seg, blk, k, TDT[dtype])
        ws = cp.alloc_workspace(prob)
        O, lse = torch.full_like(q, 7.0), torch.full(q.shape[:3], 7.0, device="cuda")
        cp.attention(prob, q, kk, v, idx[b].contiguous(), cnt[b].contiguous(), ws, O=O, lse=lse)
        assert cp.device_status(ws) == (7 if broken else 0)
        return O, lse
    O, lse = run(slice(0, items))
    for i in range(items):
        Oi, lse_i = run(slice(i, i + 1))
        assert torch.equal(O[i], Oi[0]) and torch.equal(lse[i], lse_i[0])
    assert (O == 0).all(-1).any() and bool((lse == 7).any()) == broken


@pytest.mark.parametrize("dtype", ["bf16", "f16"])
@pytest.mark.parametrize("seg,blk,k", [(384, 32, 20), (384, 128, 7), (128, 64, 9)])
def test_mixed_lists_on_the_single_cta_kernel(dtype, seg, blk, k):
    """Segments of an odd number of 128-row tiles never take pairs of CTAs."""
    Hq, Hkv, n = 4, 2, 2500
    Q, K, V = make_uniform_qkv(1, Hq, Hkv, n, 128, dtype=dtype, seed=seg + k)
    idx, cnt = mixed_lists(Hq, n, seg, blk, k, k, False)
    prob = cp.Problem(1, Hq, Hkv, n, 128, seg, blk, k, TDT[dtype])
    ws = cp.alloc_workspace(prob)
    O, lse = cp.attention(prob, Q.cuda(), K.cuda(), V.cuda(), idx.cuda(), cnt.cuda(), ws, want_lse=True)
    assert cp.device_status(ws) == 0
    O_ref, lse_ref = oracle.sparse_attention(Q, K, V, idx.numpy(), cnt.numpy(), seg, blk, SM)
    assert_close(O, O_ref, V, dtype)
    none = np.isneginf(lse_ref)
    assert none.any() and np.array_equal(np.isneginf(lse.cpu().numpy()), none)
    assert np.abs(lse.cpu().numpy()[~none] - lse_ref[~none]).max() <= 1e-4


@pytest.mark.parametrize("seg", [256, 384])
def test_a_wait_that_runs_out_is_reported(seg):
    """V tiles never requested (test hook): pairs of CTAs (segment 256) and the single-CTA kernel give up after their limit, and the next call works."""
    Q, K, V = (t.cuda() for t in make_uniform_qkv(1, 2, 1, 700, 128, seed=seg))
    out = []
    for flags, status in ((0, 0), (cp.FLAG_TEST_WITHHOLD_V, 6), (0, 0)):
        prob = cp.Problem(1, 2, 1, 700, 128, seg, 64, 8, torch.bfloat16, flags=flags)
        ws = cp.alloc_workspace(prob)
        idx, cnt = cp.select(prob, cp.estimate(prob, Q, K, ws), ws)
        out.append(cp.attention(prob, Q, K, V, idx, cnt, ws))
        assert cp.device_status(ws) == status
    assert torch.equal(out[0], out[2])
