"""Thresholds of rows whose logits are large and widely spread (supports of one or a few chunks, maxima far above the spacing
of floats near 1): every row with candidates must route at least one chunk, and its threshold must be the float64 root.

Bound: tau is 1-Lipschitz in the logits (maximum norm).  A logit is a sum of head_dim products in fp32, so it is off by at most
head_dim * 2^-24 times the sum of their magnitudes, S; the sum of powers is met within 4e-6, and its slope is at least 1;
tau itself is rounded to fp32."""
import math

import pytest
import torch

from paper_2605_18753_b200 import binding as B

pytestmark = pytest.mark.gpu
DEV = "cuda"


def _tau64(x, e):
    """Root of sum [x - tau]_+^e = 1 along the last axis, rows of -inf padding allowed (bisection in float64)."""
    high = x.amax(-1)
    low = high - 1.0
    for _ in range(60):
        mid = 0.5 * (low + high)
        above = (x - mid[..., None]).clamp(min=0.0).pow(e).sum(-1) >= 1.0
        low, high = torch.where(above, mid, low), torch.where(above, high, mid)
    return 0.5 * (low + high)


def _check(p, Q, Kbar, tau, count, n_cand, alpha):
    """Q [b, n, h_q, d], Kbar [b, h_kv, T, d], tau [b, h_q, n], count [b, h_kv, n], n_cand [b, n]."""
    g_q, scale = p.h_q // p.h_kv, p.gamma * (alpha - 1.0) / math.sqrt(p.head_dim)
    cand = torch.arange(Kbar.shape[2], device=DEV)[None, None] < n_cand[..., None]           # [b, n, T]
    some = n_cand > 0
    worst = 0.0
    for r in range(p.h_kv):
        assert (count[:, r][some] >= 1).all(), "a row with candidates routes nothing"
        for h in range(r * g_q, (r + 1) * g_q):
            q, k = Q[:, :, h].double(), Kbar[:, r].double()
            x = (torch.einsum("bnd,btd->bnt", q, k) * scale).masked_fill(~cand, -math.inf)
            S = (torch.einsum("bnd,btd->bnt", q.abs(), k.abs()) * scale).masked_fill(~cand, 0.0).amax(-1)
            want = torch.where(some, _tau64(x, 1.0 / (alpha - 1.0)), 0.0)
            tol = p.head_dim * 2.0 ** -24 * S + 4e-6 + 2.0 ** -23 * want.abs()
            err = (tau[:, h].double() - want).abs()
            assert torch.isfinite(tau[:, h]).all()
            assert (err[some] <= tol[some]).all(), float((err - tol)[some].max())
            worst = max(worst, float(err[some].max()))
    return worst


def _inputs(batch, n, h_q, h_kv, d, T, spread, offset, dtype, seed):
    """Logits (at gamma = 1 / (alpha - 1)) of deviation about `spread` around `offset`."""
    g = torch.Generator(DEV).manual_seed(seed)
    u = torch.randn(d, generator=g, device=DEV)
    u /= u.norm()
    Q = (torch.randn(batch, n, h_q, d, generator=g, device=DEV) + math.sqrt(d) * u).to(dtype)
    Kbar = spread * torch.randn(batch, h_kv, T, d, generator=g, device=DEV) + offset * u
    return Q, Kbar


@pytest.mark.parametrize("alpha", [1.25, 1.5, 2.0, 1.75])
@pytest.mark.parametrize("spread,offset", [(3.0, 40.0), (16.0, 0.0), (32.0, -40.0), (300.0, 0.0)])
@pytest.mark.parametrize("kw", [
    dict(n=2000, h_q=4, h_kv=1, head_dim=64, block=16, dtype=torch.bfloat16),          # up to 125 candidates: held in registers; streamed where a tile spans chunks
    dict(n=16 * 620, h_q=8, h_kv=1, head_dim=64, block=16, dtype=torch.bfloat16),      # streamed, three threads per row, clusters of two
    dict(n=1500, h_q=2, h_kv=2, head_dim=128, block=16, dtype=torch.bfloat16),         # one query head per KV head
    dict(n=16 * 140, h_q=2, h_kv=1, head_dim=64, block=16, dtype=torch.float32),       # CUDA cores
    dict(n=800, h_q=2, h_kv=1, head_dim=64, block=16, dtype=torch.float32, causal=0),
])
def test_prefill_thresholds(alpha, spread, offset, kw):
    kw = dict(kw)
    n, block, dtype, causal = kw.pop("n"), kw.pop("block"), kw.pop("dtype"), kw.pop("causal", 1)
    d = kw["head_dim"]
    p = B.make_params(batch=1, seq_q=n, seq_kv=n, block=block, dtype=dtype, alpha=alpha, gamma=1.0 / (alpha - 1.0), causal=causal, **kw)
    Q, Kbar = _inputs(1, n, p.h_q, p.h_kv, d, n // block, spread, offset, dtype, seed=int(spread) + n)
    ws, rt = B.alloc_workspace(p), B.alloc_routing(p, with_tau=True)
    B.dash_attn_select(p, Q, Kbar, rt["mask"], rt["count"], rt["blk_idx"], rt["blk_bias"], ws, tau=rt["tau"])
    assert B.dash_attn_last_status(ws) == 0
    n_cand = torch.arange(n, device=DEV)[None] // block if causal else torch.full((1, n), n // block, device=DEV)
    _check(p, Q, Kbar, rt["tau"], rt["count"], n_cand, alpha)


@pytest.mark.parametrize("alpha", [1.25, 1.5, 2.0, 1.75])
@pytest.mark.parametrize("spread,offset", [(3.0, 40.0), (16.0, 0.0), (32.0, -40.0), (300.0, 0.0)])
@pytest.mark.parametrize("T,lens", [(64, [64, 64, 30]), (512, [512, 300, 129]), (2200, [2200, 2049, 600])])
def test_decode_thresholds(alpha, spread, offset, T, lens):
    block, d, batch = 16, 64, 8                      # (many rows: the start depends on the row)
    lens = [lens[i % 3] * block - i for i in range(batch)]
    p = B.make_params(batch=batch, seq_q=1, seq_kv=T * block, h_q=8, h_kv=2, head_dim=d, block=block, dtype=torch.bfloat16,
                      alpha=alpha, gamma=1.0 / (alpha - 1.0))
    Q, Kbar = _inputs(batch, 1, 8, 2, d, T, spread, offset, torch.bfloat16, seed=T + int(spread))
    kv_len = torch.tensor(lens, dtype=torch.int32, device=DEV)
    ws, rt = B.alloc_workspace(p), B.alloc_routing(p, with_tau=True)
    B.dash_attn_select(p, Q[:, 0].contiguous(), Kbar, rt["mask"], rt["count"], rt["blk_idx"], rt["blk_bias"], ws, tau=rt["tau"],
                       kv_len=kv_len)
    assert B.dash_attn_last_status(ws) == 0
    _check(p, Q, Kbar, rt["tau"], rt["count"], ((kv_len - 1) // block)[:, None].long(), alpha)
