"""dK and dV of the two-term backward carry the rounding of the weights (two bf16 terms: 2^-17 at most, each) and nothing that
grows with the length: sums of many query tiles, several heads per KV head, against float64 on the same routing."""
import math

import pytest
import torch

from paper_2605_18753_b200 import binding as B
from paper_2605_18753_b200 import synth
from tests.test_gpu_parity import _wl

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("seq,h_q,h_kv,head_dim,block", [(3000, 16, 1, 64, 64), (3000, 32, 2, 64, 128), (2500, 16, 1, 128, 64), (2000, 8, 1, 128, 32),
                                                         (1500, 2, 2, 64, 16), (130, 4, 1, 64, 64)])
def test_sums_do_not_lose_bits_with_the_length(seq, h_q, h_kv, head_dim, block):
    # (a small temperature: every candidate is routed, so a row's list is its chunks in order)
    w = _wl(seq=seq, h_q=h_q, h_kv=h_kv, head_dim=head_dim, block=block, gamma=0.05, sigma=1.0, seed=77)
    inp = synth.make_prefill_inputs(w, DEV)
    Q, K, V = inp["Q"], inp["K"], inp["V"]
    dO = torch.randn(Q.shape, device=DEV, generator=torch.Generator(DEV).manual_seed(78)).to(Q.dtype)
    p = B.params_for_prefill(Q, K, V, dO, block=block, alpha=w.alpha, gamma=w.gamma, sigma=w.sigma)
    ws, kbar, rt = B.alloc_workspace(p), B.alloc_kbar(p), B.alloc_routing(p)
    B.dash_attn_block_summaries(p, K, kbar)
    B.dash_attn_select(p, Q, kbar, rt["mask"], rt["count"], rt["blk_idx"], rt["blk_bias"], ws)
    row = torch.arange(seq, device=DEV)
    own = row // block
    assert (rt["count"][0] == own[None]).all()
    dQ, dK = torch.empty_like(Q), torch.empty(1, seq, h_kv, head_dim, device=DEV)
    dV, db = torch.empty_like(dK), torch.empty_like(rt["blk_bias"])
    B.dash_attn_bwd_attend_prefill(p, Q, K, V, dO, rt["mask"], rt["blk_bias"], dQ, dK, dV, db)
    g, scale = h_q // h_kv, 1.0 / math.sqrt(head_dim)
    for r in range(h_kv):
        at = torch.tensor([B.dash_attn_list_offset(p, 0, r, i) for i in range(seq)], device=DEV)[:, None] + own[None]
        bias = torch.where(own[None] < own[:, None], rt["blk_bias"][at.clamp(max=db.numel() - 1)].double(), 0.0)
        bias = bias.masked_fill(row[None] > row[:, None], -math.inf)
        want_k = want_v = 0.0
        for h in range(r * g, (r + 1) * g):
            q, k, v, do = Q[0, :, h].double(), K[0, :, r].double(), V[0, :, r].double(), dO[0, :, h].double()
            P = torch.softmax(q @ k.T * scale + bias, -1)
            dP = do @ v.T
            dS = P * (dP - (P * dP).sum(-1, keepdim=True))
            want_k, want_v = want_k + dS.T @ q * scale, want_v + P.T @ do
        for got, want, name in ((dK[0, :, r], want_k, "dK"), (dV[0, :, r], want_v, "dV")):
            err = float((got.double() - want).norm() / want.norm())
            assert err <= 2.0 ** -17, (name, err)
