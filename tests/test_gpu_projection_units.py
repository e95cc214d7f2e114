"""The projection's unit schedule: fewer query units than SMs, a last round that is nearly empty, segments of one and of many
tiles, ragged lengths, with and without values.  Q, K, V against plain fp32 products; the representatives left in the workspace
against a pass over the stored Q and K (scores with and without it are the same bits)."""
import dataclasses

import pytest
import torch

from paper_2409_12490_b200 import binding as cp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("values", [True, False])
@pytest.mark.parametrize("B,n,seg,blk,Hq,Hkv", [(1, 128, 128, 32, 2, 2), (1, 2000, 1024, 128, 4, 2), (2, 1300, 512, 64, 16, 4),
                                                (1, 4500, 128, 32, 8, 8), (1, 1153, 256, 128, 3, 1),
                                                (1, 3301, 256, 64, 32, 8), (1, 300, 512, 64, 32, 8)])
def test_every_tile_is_projected_once(B, n, seg, blk, Hq, Hkv, values):
    torch.manual_seed(n)
    D, dm = 128, 256
    mk = lambda *s: torch.randn(*s, device="cuda").to(torch.bfloat16)
    X, Wq, Wk, Wv = mk(B, n, dm), mk(Hq * D, dm) / 16, mk(Hkv * D, dm) / 16, mk(Hkv * D, dm) / 16
    prob = cp.Problem(B, Hq, Hkv, n, D, seg, blk, seg // blk + 2, torch.bfloat16)
    ws = cp.alloc_workspace(prob)
    poison = lambda h: torch.full((B, h, n, D), float("nan"), dtype=torch.bfloat16, device="cuda")
    if values:
        Q, K, V = cp.project_qkv(prob, X, Wq, Wk, Wv, ws, Q_out=poison(Hq), K_out=poison(Hkv), V_out=poison(Hkv))
    else:
        Q, K = cp.project_qk(prob, X, Wq, Wk, ws, Q_out=poison(Hq), K_out=poison(Hkv))
    S = cp.estimate(dataclasses.replace(prob, flags=cp.FLAG_SUMMARIES_READY), Q, K, ws)
    assert cp.device_status(ws) == 0
    torch.backends.cuda.matmul.allow_tf32 = False
    for got, W, h in ((Q, Wq, Hq), (K, Wk, Hkv)) + (((V, Wv, Hkv),) if values else ()):
        ref = (X.double() @ W.double().T).view(B, n, h, D).permute(0, 2, 1, 3)
        # one rounding to bf16 (2^-8) of a sum of 256 products accumulated in fp32
        assert ((got.double() - ref).abs() <= 2.0 ** -8 * ref.abs() + 1e-4).all()
    assert torch.equal(S, cp.estimate(prob, Q, K, cp.alloc_workspace(prob)))
