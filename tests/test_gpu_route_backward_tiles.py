"""The routing backward where sixteen tokens share a block, and on either side of the line to the warp-per-row kernel (lists longer
than fit in shared memory; sixteen heads): dQ and dKbar against float64 on the library's lists and thresholds.  A small
temperature (alpha = 2, whose margins are 1 / n, needs a smaller one) routes every candidate, with margins of about n^(-1/2), so that the Jacobian is well conditioned: logits carry
fp32-class errors (2e-6), a margin of 1/30 turns them into 1e-4 of the weights, and differences against the mean double that."""
import math

import pytest
import torch

from paper_2605_18753_b200 import binding as B
from paper_2605_18753_b200 import synth
from tests.test_gpu_parity import _wl

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("alpha", [1.5, 2.0])
@pytest.mark.parametrize("seq,block,h_q,h_kv,head_dim,batch,local", [
    (17, 16, 4, 2, 64, 1, 0), (130, 16, 4, 4, 128, 2, 0), (1003, 32, 8, 2, 64, 2, 1), (700, 64, 16, 2, 128, 1, 0),
    (2960, 16, 4, 1, 128, 1, 0), (3008, 16, 4, 1, 128, 1, 0),         # 184 chunks, the last that fit, and 188
    (500, 32, 16, 1, 64, 1, 0),
])
def test_gradients_through_the_routing(alpha, seq, block, h_q, h_kv, head_dim, batch, local):
    w = _wl(seq=seq, h_q=h_q, h_kv=h_kv, head_dim=head_dim, block=block, alpha=alpha, gamma=0.05 if alpha < 2.0 else 0.005, sigma=2.0, seed=71, batch=batch)
    inp = synth.make_prefill_inputs(w, DEV)
    Q, K = inp["Q"], inp["K"]
    p = B.params_for_prefill(Q, K, inp["V"], Q, block=block, alpha=alpha, gamma=w.gamma, sigma=w.sigma, local_blocks=local)
    ws, kbar, rt = B.alloc_workspace(p), B.alloc_kbar(p), B.alloc_routing(p, with_tau=True)
    B.dash_attn_block_summaries(p, K, kbar)
    B.dash_attn_select(p, Q, kbar, rt["mask"], rt["count"], rt["blk_idx"], rt["blk_bias"], ws, tau=rt["tau"])
    dbias = torch.randn(rt["blk_bias"].shape, device=DEV, generator=torch.Generator(DEV).manual_seed(72))
    dQ, dKbar = torch.empty(Q.shape, device=DEV), torch.empty_like(kbar)
    B.dash_attn_bwd_select_prefill(p, Q, kbar, rt["count"], rt["blk_idx"], rt["tau"], dbias, dQ, dKbar)
    g, e, T = h_q // h_kv, 1.0 / (alpha - 1.0), seq // block
    row, chunk = torch.arange(seq, device=DEV), torch.arange(T, device=DEV)
    own = row // block
    n = (own - local).clamp(min=0)                                      # every candidate is routed, in order
    on = chunk[None] < n[:, None]
    for b in range(batch):
        for r in range(h_kv):
            assert (rt["count"][b, r] == torch.minimum(own, n + local)).all()
            at = torch.tensor([B.dash_attn_list_offset(p, b, r, i) for i in range(seq)], device=DEV)[:, None] + chunk[None]
            db = torch.where(on, dbias[at.clamp(max=dbias.numel() - 1)].double(), 0.0)
            q, kb = Q[b, :, r * g:(r + 1) * g].double(), kbar[b, r].double()
            scale = w.gamma / math.sqrt(head_dim)
            m = torch.einsum("nhd,td->nht", q, kb) * (scale * (alpha - 1.0)) - rt["tau"][b, r * g:(r + 1) * g].T[..., None].double()
            m = torch.where(on[:, None], m.clamp(min=0.0), 0.0)
            weight = m.pow(e).mean(1)
            dp = torch.where(on, (db - db.sum(1, keepdim=True) / n.clamp(min=1)[:, None]) / w.sigma / weight.clamp(min=1e-300) / g, 0.0)[:, None]
            s = torch.where(m > 0, m.clamp(min=1e-300).pow(e - 1.0), 0.0)
            dz = s * (dp - (s * dp).sum(2, keepdim=True) / s.sum(2, keepdim=True).clamp(min=1e-300)) * scale
            for got, want in ((dQ[b, :, r * g:(r + 1) * g], torch.einsum("nht,td->nhd", dz, kb)), (dKbar[b, r], torch.einsum("nht,nhd->td", dz, q))):
                err = float((got.double() - want).norm() / want.norm().clamp(min=1e-30))
                assert err <= 2e-4, err
