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


@pytest.mark.parametrize("dtype,B,Hkv,g,n,seg,blk", [
    ("bf16", 1, 8, 4, 6000, 256, 16),          # parts that begin inside a row group, 375 blocks
    ("f16", 1, 2, 4, 8192, 128, 32),           # whole row groups of 16 segments
    ("bf16", 2, 3, 1, 4097, 64, 64),           # single heads, a last row group of one segment
    ("f16", 1, 2, 2, 2050, 32, 32),
])
@pytest.mark.parametrize("fuse", [False, True])
def test_marks_anywhere(dtype, B, Hkv, g, n, seg, blk, fuse):
    """Values that do not fit in single rows and blocks, in all blocks of a tile, in all rows of a row group."""
    Q, K, _ = make_uniform_qkv(B, Hkv * g, Hkv, n, 128, dtype=dtype, seed=n)
    small = 3e-8 if dtype == "bf16" else 6e-8
    rng = np.random.default_rng(n)
    if dtype == "f16":                         # 2^-24 does not fit beside these
        Q[..., 3] = 80.0
        K[..., 3] = -80.0
    for b in range(B):
        for h in range(Hkv * g):
            for j in rng.choice(-(-n // seg), 3):
                Q[b, h, j * seg:(j + 1) * seg, 7] = small
        for h in range(Hkv):
            for x in rng.choice(-(-n // blk), 9):
                K[b, h, x * blk:(x + 1) * blk, rng.integers(8, 128)] = -small
    K[:, :, 32 * blk:64 * blk, 11] = small     # the second tile of every row group
    Q[0, :g, :(64 if g == 1 else 32 if g == 2 else 16) * seg, 90] = small
    check(Q, K, dtype, seg, blk, est_scale=0.01, fuse=fuse)


def test_marks_of_more_tiles_than_are_kept():
    """A CTA's share of some 880 tiles, of which the marks of the last 512 are kept; sampled rows against fp64."""
    Hq, Hkv, n, blk = 8, 1, 131072, 16
    g = torch.Generator(device="cuda").manual_seed(11)
    Q, K = (torch.randn(1, h, n, 128, generator=g, device="cuda").to(torch.bfloat16) for h in (Hq, Hkv))
    n2 = n // blk
    marked = torch.rand(n2, generator=g, device="cuda") < 0.02
    K[0, 0, :, 5] = torch.where(marked.repeat_interleave(blk), torch.full((n,), 3e-8, device="cuda"), K[0, 0, :, 5].float()).to(K.dtype)
    rows = [(h, j) for h in (0, 3, 7) for j in (1, 100, 2047, 4096, 6001, 8190, 8191)]
    for h, j in rows[::2]:
        Q[0, h, j * blk:(j + 1) * blk, 6] = 3e-8
    prob = cp.Problem(1, Hq, Hkv, n, 128, blk, blk, 4, torch.bfloat16, est_scale=0.1)
    ws = cp.alloc_workspace(prob)
    S = cp.estimate(prob, Q, K, ws)
    assert cp.device_status(ws) == 0
    rep = lambda X: (X.view(X.shape[0], -1, blk, 128).amax(2).double(), X.view(X.shape[0], -1, blk, 128).amin(2).double())
    (Qmax, Qmin), (Kmax, Kmin) = rep(Q[0]), rep(K[0])
    for h, j in rows:
        l = [q[h, j] @ k[0].T * f32(0.1) for q in (Qmax, Qmin) for k in (Kmax, Kmin)]
        l = [x - x.logsumexp(0) for x in l]
        ref = torch.maximum(torch.logaddexp(l[0], l[2]), torch.logaddexp(l[1], l[3])) - np.log(2.0)
        ref[j + 1:] = float("-inf")
        assert torch.equal(torch.isneginf(S[0, h, j]), torch.isneginf(ref))
        assert (S[0, h, j, :j + 1] - ref[:j + 1]).abs().max().item() <= 1e-9


def score_times(dtype, change):
    """us of both score kernels at 65536 tokens, 32 / 8 heads, segment 512, block 64, without and with a change to Q and K."""
    Hq, Hkv, n, seg, blk = 32, 8, 65536, 512, 64
    g = torch.Generator(device="cuda").manual_seed(7)
    Q, K = (torch.randn(1, h, n, 128, generator=g, device="cuda").to(DT[dtype]) for h in (Hq, Hkv))
    out = []
    for f in (lambda: None, lambda: change(Q, K, seg, blk)):
        f()
        prob = cp.Problem(1, Hq, Hkv, n, 128, seg, blk, 16, DT[dtype])
        ws = cp.alloc_workspace(prob)
        S = cp.estimate(prob, Q, K, ws)
        prob.flags = cp.FLAG_SUMMARIES_READY
        times = []
        for _ in range(9):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record()
            for _ in range(4):
                cp.estimate(prob, Q, K, ws, S_out=S)
            b.record()
            torch.cuda.synchronize()
            times.append(a.elapsed_time(b))
        out.append(sorted(times)[4] * 250)
        assert cp.device_status(ws) == 0
    return out


def one_row(Q, K, seg, blk):
    Q[0, 5, 40 * seg:41 * seg, 9] = 3e-8                       # one of the 8192 query representatives' segments


def some_blocks(Q, K, seg, blk):
    for i in range(0, K.shape[2] // blk, 20):                  # 5 % of the blocks of every head
        K[0, :, i * blk:(i + 1) * blk, 77] = 3e-8


def everything(Q, K, seg, blk):
    Q[..., 3] = 3e-8
    K[..., 3] = 3e-8


# Both kernels of the scores, with / without: 183, 190 and 272 us against 176; with marked logits summed by single threads 225, 229 and 1641.
# Times of a shared machine, hence the room.
@pytest.mark.parametrize("change,limit", [(one_row, 1.15), (some_blocks, 1.2), (everything, 2.5)])
def test_values_that_do_not_fit_cost_little(change, limit):
    plain, marked = score_times("bf16", change)
    print(f"{change.__name__}: {plain:.0f} us, marked {marked:.0f} us")
    assert marked < limit * plain
