"""The selection kernel on score rows that its search can go wrong on: row lengths around the number of ranked candidates, of
warps' parts and of keys per thread; scores in one bin of a digit, equal scores, infinities, both zeros, values beyond the range that
the first digit spreads.  Exact against the oracle's full sort."""
import numpy as np
import pytest
import torch

import oracle
from paper_2409_12490_b200 import binding as cp

pytestmark = pytest.mark.gpu


def rows(n, rng):
    """One score row per kind, [kinds, n] float64."""
    normal = rng.standard_normal(n)
    kinds = [
        -30.0 + 12.0 * normal,                                       # as ln S is distributed
        np.full(n, -7.25),                                           # all equal: by index alone
        np.where(rng.random(n) < 0.05, -5.0 * rng.random(n), -np.inf),
        -1.0 - 1e-13 * rng.integers(0, 50, n),                       # differ in the last bytes only, with ties
        np.round(4.0 * normal) / 4.0,                                # both signs, both zeros, many ties
        -1e5 - 1e4 * rng.random(n),                                  # below the first digit's range
        -1e-3 * rng.random(n),                                       # above it
        np.where(rng.random(n) < 0.5, -0.0, 0.0),
        np.where(rng.random(n) < 0.3, -20.0, -20.0 - normal ** 2),   # a tie that reaches across the threshold
        np.exp(200.0 * normal) * np.where(rng.random(n) < 0.5, -1.0, 1.0),
    ]
    return np.stack(kinds)


@pytest.mark.parametrize("n2", [2, 33, 128, 129, 130, 257, 1000, 1024, 1025, 2050, 4096, 4097, 8192])
def test_one_row_per_head(n2):
    rng = np.random.default_rng(n2)
    S = rows(n2, rng)
    H = S.shape[0]
    for k in sorted({1, 2, min(65, n2 - 1), n2 // 2, n2 - 1} - {0}):
        prob = cp.Problem(1, H, H, 16 * n2, 64, 16, 16, k, torch.bfloat16)
        ws = cp.alloc_workspace(prob)
        idx, cnt = cp.decode_select(prob, torch.from_numpy(S[None]).cuda(), ws)
        idx_ref, cnt_ref = oracle.decode_select(S[None], k)
        assert np.array_equal(cnt.cpu().numpy(), cnt_ref), k
        assert np.array_equal(idx.cpu().numpy(), idx_ref), k


@pytest.mark.parametrize("n2,r,k,group,n_sink,n_local", [(300, 8, 20, 1, 0, 0), (701, 4, 140, 5, 0, 0), (520, 16, 24, 2, 3, 4), (1100, 32, 300, 1, 0, 200)])
def test_segments_pools_and_forced_blocks(n2, r, k, group, n_sink, n_local):
    rng = np.random.default_rng(n2)
    n1 = -(-n2 // r)
    S = np.stack([rows(n2, rng) for _ in range(n1)], axis=1)[None]            # [1, kinds, n1, n2]
    H = S.shape[1]
    prob = cp.Problem(1, H, H // group, 16 * n2, 64, 16 * r, 16, k, torch.bfloat16, n_sink=n_sink, n_local=n_local,
                      flags=cp.FLAG_SHARED_GROUP_LISTS if group > 1 else 0)
    ws = cp.alloc_workspace(prob)
    idx, cnt = cp.select(prob, torch.from_numpy(S).cuda(), ws)
    idx_ref, cnt_ref = oracle.select(S, 16 * r, 16, k, group=group, n_sink=n_sink, n_local=n_local)
    assert np.array_equal(cnt.cpu().numpy(), cnt_ref)
    assert np.array_equal(idx.cpu().numpy(), idx_ref)
