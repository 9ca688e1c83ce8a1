"""dK and dV where a key slice gathers the tokens that attend it: group sizes from 1 to 16 (128 to 8 tokens a step), slices that only their
own chunks' tokens attend, last steps that are filled up, chunks beyond the first mask word, several blocks per slice; all four
gradients against float64 on the library's sparse routing.  Two-term products carry 2^-17 of every weight, dbias is formed in
fp32 (8e-6: sums of a few dozen terms that cancel); dQ is stored in bf16 (2^-8 at most, 2^-9 on average)."""
import math

import pytest
import torch

from paper_2605_18753_b200 import binding as B
from paper_2605_18753_b200 import synth
from tests.test_gpu_parity import _wl

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("seq,h_q,h_kv,head_dim,block,local,gamma", [
    (70, 4, 4, 64, 16, 0, 2.0), (1100, 2, 2, 64, 32, 0, 2.0), (1100, 4, 4, 128, 16, 1, 4.0), (900, 4, 2, 128, 64, 0, 4.0),
    (2400, 8, 2, 64, 64, 0, 8.0), (2431, 8, 2, 128, 128, 0, 2.0), (1000, 16, 2, 64, 16, 0, 4.0), (1300, 16, 1, 128, 32, 1, 2.0), (64, 8, 1, 64, 64, 0, 1.0),
])
def test_gathered_rows_against_float64(seq, h_q, h_kv, head_dim, block, local, gamma):
    w = _wl(seq=seq, h_q=h_q, h_kv=h_kv, head_dim=head_dim, block=block, gamma=gamma, sigma=1.0, seed=61)
    inp = synth.make_prefill_inputs(w, DEV)
    Q, K, V = inp["Q"], inp["K"], inp["V"]
    dO = torch.randn(Q.shape, device=DEV, generator=torch.Generator(DEV).manual_seed(62)).to(Q.dtype)
    p = B.params_for_prefill(Q, K, V, dO, block=block, alpha=w.alpha, gamma=w.gamma, sigma=w.sigma, local_blocks=local)
    ws, kbar, rt = B.alloc_workspace(p), B.alloc_kbar(p), B.alloc_routing(p)
    B.dash_attn_block_summaries(p, K, kbar)
    B.dash_attn_select(p, Q, kbar, rt["mask"], rt["count"], rt["blk_idx"], rt["blk_bias"], ws)
    dQ, dK = torch.empty_like(Q), torch.empty(1, seq, h_kv, head_dim, device=DEV)
    dV, db = torch.empty_like(dK), torch.empty_like(rt["blk_bias"])
    B.dash_attn_bwd_attend_prefill(p, Q, K, V, dO, rt["mask"], rt["blk_bias"], dQ, dK, dV, db)
    g, scale, T = h_q // h_kv, 1.0 / math.sqrt(head_dim), -(-seq // block)
    row, chunk = torch.arange(seq, device=DEV), torch.arange(T, device=DEV)
    own = row // block
    sq = {k: [0.0, 0.0] for k in ("dQ", "dK", "dV", "dbias")}

    def add(key, got, want):
        sq[key][0] += float((got.double() - want).pow(2).sum())
        sq[key][1] += float(want.pow(2).sum())

    for r in range(h_kv):
        bits = (rt["mask"][0, r][:, chunk // 32].long() >> (chunk % 32)[None]) & 1
        routed = (bits == 1) & (chunk[None] < own[:, None])
        at = torch.tensor([B.dash_attn_list_offset(p, 0, r, i) for i in range(seq)], device=DEV)[:, None] + routed.cumsum(1) - 1
        at = at.clamp(0, max(db.numel() - 1, 0))
        bias = torch.where(routed, rt["blk_bias"][at].double(), -math.inf) if db.numel() else torch.full((seq, T), -math.inf, dtype=torch.double, device=DEV)
        bias = torch.where(chunk[None] == own[:, None], 0.0, bias)[:, own]
        bias = bias.masked_fill(row[None] > row[:, None], -math.inf)
        want_k = want_v = want_b = 0.0
        for h in range(r * g, (r + 1) * g):
            q, k, v, do = Q[0, :, h].double(), K[0, :, r].double(), V[0, :, r].double(), dO[0, :, h].double()
            P = torch.softmax(q @ k.T * scale + bias, -1)
            dP = do @ v.T
            dS = P * (dP - (P * dP).sum(-1, keepdim=True))
            add("dQ", dQ[0, :, h], dS @ k * scale)
            want_k, want_v = want_k + dS.T @ q * scale, want_v + P.T @ do
            want_b = want_b + torch.zeros(seq, T, dtype=torch.double, device=DEV).index_add(1, own, dS)
        add("dK", dK[0, :, r], want_k)
        add("dV", dV[0, :, r], want_v)
        if routed.any():
            add("dbias", db[at][routed], want_b[routed])
    for key, bound in (("dQ", 2.0 ** -8), ("dK", 2.0 ** -17), ("dV", 2.0 ** -17), ("dbias", 8e-6)):
        err, norm = (math.sqrt(x) for x in sq[key])
        assert err <= bound * norm, (key, err / max(norm, 1e-300))
