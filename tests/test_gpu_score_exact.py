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


def signed_bytes(x):
    """The four signed bytes of integers of 31 bits, lowest first."""
    out = []
    for _ in range(4):
        d = (x + 128) % 256 - 128
        out.append(d)
        x = (x - d) // 256
    assert not x.any()
    return out


@pytest.mark.parametrize("dtype", ["bf16", "f16"])
@pytest.mark.parametrize("shift,decisive", [(0, {0, 1, 2}), (8, {2, 3, 4}), (12, {2, 3, 4}), (18, {4, 5, 6})])
def test_every_accumulator_decides(dtype, shift, decisive):
    """Odd multiples of 2^(shift - 24) of both signs beside a 32 that meets a 0: the bytes that hold them carry the logits."""
    Hq, Hkv, n1, r, blk = 8, 2, 40, 2, 16
    rng = np.random.default_rng(shift)
    bits = 8 if dtype == "bf16" else 11
    odd = lambda *size: (2 * rng.integers(0, 2 ** (bits - 1), size) + 1) * rng.choice([-1, 1], size) * 2 ** shift
    q, k = odd(1, Hq, n1, 128), odd(1, Hkv, n1 * r, 128)
    q[..., 0], q[..., 1], k[..., 0], k[..., 1] = 0, 2 ** 29, 2 ** 29, 0
    Q, K = (torch.from_numpy(x * 2.0 ** -24).to(DT[dtype]) for x in (q, k))
    assert np.array_equal(Q.double().numpy() * 2 ** 24, q) and np.array_equal(K.double().numpy() * 2 ** 24, k)
    est_scale = 2.0 ** (48 - 2 * (shift + bits) + 1)                           # logits of the order of ten
    qd, kd = signed_bytes(q), signed_bytes(k.repeat(Hq // Hkv, axis=1))
    acc = [sum(qd[i] @ kd[s - i].swapaxes(-1, -2) for i in range(max(0, s - 3), min(s, 3) + 1)) for s in range(7)]
    part = [np.abs(a).max() * 2.0 ** (8 * s - 48) * est_scale for s, a in enumerate(acc)]
    assert {s for s in range(7) if part[s] > 1e-5} >= decisive, part
    check(Q.repeat_interleave(r * blk, 2), K.repeat_interleave(blk, 2), dtype, r * blk, blk, est_scale=est_scale)


@pytest.mark.parametrize("power", [-64, 70])
@pytest.mark.parametrize("which", ["Q", "K", "both"])
def test_magnitudes_beyond_the_scales(power, which):
    """bf16 rows or blocks whose exponent is out of range: marked, with logits of the usual size."""
    Q, K, _ = make_uniform_qkv(1, 8, 2, 1500, 128, seed=9)
    if which != "K":
        Q = (Q.float() * 2.0 ** power).bfloat16()
    if which != "Q":
        K = (K.float() * 2.0 ** (-power if which == "both" else power)).bfloat16()
    check(Q, K, "bf16", 128, 32, est_scale=0.125 * (1.0 if which == "both" else 2.0 ** -power))


def maps(Q, K, seg, blk):
    """The four logit maps of Algorithm 1; a NaN is left out of a maximum or minimum."""
    rep = lambda X, size: [[f([X[:, :, i:i + size]], axis=3)[0] for i in range(0, X.shape[2], size)] for f in (np.fmax.reduce, np.fmin.reduce)]
    q, k = [[np.stack(x, 2) for x in rep(X.double().numpy(), size)] for X, size in ((Q, seg), (K, blk))]
    k = [x.repeat(Q.shape[1] // K.shape[1], axis=1).swapaxes(-1, -2) for x in k]
    with np.errstate(invalid="ignore"):
        return [a @ b for a in q for b in k]


@pytest.mark.parametrize("dtype", ["bf16", "f16"])
@pytest.mark.parametrize("where", ["Q", "K", "future", "several"])
@pytest.mark.parametrize("value", [float("inf"), float("-inf")])
def test_infinities(dtype, where, value):
    """A map of a row with an infinite logit has no log-sum-exp: the row's scores follow from its other maps.  Rows without one, and blocks that such
    maps rule out, as ever."""
    Q, K, _ = make_uniform_qkv(1, 8, 2, 2500, 128, dtype=dtype, seed=3)
    if where in ("Q", "several"):
        Q[0, 3, 700, 5] = Q[0, 1, 1300, 100] = value
    if where in ("K", "several"):
        K[0, 1, 333, 5] = value
    if where == "future":
        K[0, 1, 2499, 5] = value
    prob = cp.Problem(1, 8, 2, 2500, 128, 128, 32, 4, DT[dtype], est_scale=0.25, flags=cp.FLAG_FORCE_SPLIT_SCORE)
    ws = cp.alloc_workspace(prob)
    S = cp.estimate(prob, Q.cuda(), K.cuda(), ws).cpu().numpy()
    assert cp.device_status(ws) == 0
    L = []
    for l in maps(Q, K, 128, 32):
        l = 0.25 * l
        m = l.max(-1, keepdims=True)
        with np.errstate(invalid="ignore"):
            L.append(np.where(np.isfinite(m), l - m - np.log(np.exp(l - m).sum(-1, keepdims=True)), np.nan))
    with np.errstate(invalid="ignore"):
        pair = lambda a, b: np.where(np.isnan(a), b, np.where(np.isnan(b), a, np.logaddexp(a, b) - np.log(2.0)))
    ref = np.fmax(pair(L[0], L[2]), pair(L[1], L[3]))
    masked = oracle.estimation.causal_block_mask(20, 79, 128, 32)
    assert any(np.isnan(x).any() for x in L) and np.isneginf(S[..., masked]).all()
    assert np.isfinite(ref[..., ~masked]).all() and np.abs(S - ref)[..., ~masked].max() <= 1e-9


@pytest.mark.parametrize("dtype", ["bf16", "f16"])
@pytest.mark.parametrize("where", ["Q", "K", "tokens", "S_prev nan", "S_prev inf", "S_prev -inf"])
def test_not_finite_as_in_the_general_kernel(dtype, where):
    """Single NaN in Q or K (left out of the representatives) and S' that is not finite: both paths agree."""
    Q, K, _ = make_uniform_qkv(1, 8, 2, 2500, 128, dtype=dtype, seed=4)
    Q0, K0, _ = make_uniform_qkv(1, 8, 2, 2500, 128, dtype=dtype, seed=5)
    if where == "Q":
        Q[0, 3, 700, 5] = Q[0, 1, 1300:1310] = float("nan")
    if where == "K":
        K[0, 1, 333, 5] = K[0, 0, 2499, 7] = float("nan")
    if where == "tokens":
        K[0, :, 64:90] = Q[0, 2, 128:200] = float("nan")
    out = []
    for flags in (0, cp.FLAG_FORCE_SPLIT_SCORE):
        prob = cp.Problem(1, 8, 2, 2500, 128, 128, 32, 4, DT[dtype], est_scale=0.25, flags=flags)
        ws = cp.alloc_workspace(prob)
        S_prev = cp.estimate(prob, Q0.cuda(), K0.cuda(), ws)
        if where.startswith("S_prev"):
            S_prev[0, 2, 10:14, 3:9] = float(where.split()[1])
        S = cp.estimate(prob, Q.cuda(), K.cuda(), ws, S_prev=S_prev)
        assert cp.device_status(ws) == 0
        out.append(S.cpu().numpy())
    a, b = out
    assert all(np.array_equal(f(a), f(b)) for f in (np.isnan, np.isposinf, np.isneginf))
    finite = np.isfinite(a)
    assert np.abs(a[finite] - b[finite]).max() <= 1e-9


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
# Times vary from run to run, hence the room.
@pytest.mark.parametrize("change,limit", [(one_row, 1.15), (some_blocks, 1.2), (everything, 2.5)])
def test_values_that_do_not_fit_cost_little(change, limit):
    plain, marked = score_times("bf16", change)
    print(f"{change.__name__}: {plain:.0f} us, marked {marked:.0f} us")
    assert marked < limit * plain
