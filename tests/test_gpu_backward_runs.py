"""dK and dV where a key slice takes runs of neighbouring tokens as they are, because most of them attend it, beside runs that it gathers:
masks from a few chunks to all of them, and both in turn, so that a run under way has to make room, at group sizes from 1 to 16
(runs of 32, 16 and 8 tokens, one to four of them a step), lengths that cut the last run, several blocks per slice.  dQ and dbias
come from the same lists.  Against float64: two-term products carry 2^-17 of every weight, one-term ones 2^-8 (dK, dV of the
tensor-core entry point), dbias is formed in fp32 (8e-6, see test_gpu_backward_gather), dQ is stored in bf16."""
import math

import pytest
import torch

from paper_2605_18753_b200 import binding as B

pytestmark = pytest.mark.gpu
DEV = "cuda"


def _routing(p, n, h_kv, block, pattern, gen):
    """Mask, lists and biases of random rows: every earlier chunk with a probability that depends on the row."""
    T, words = -(-n // block), (-(-n // block) + 31) // 32
    row, chunk = torch.arange(n, device=DEV), torch.arange(T, device=DEV)
    own = row // block
    share = {"few": torch.full((n,), 0.06), "most": torch.full((n,), 0.9), "all": torch.ones(n),
             "turns": torch.where((torch.arange(n) // 40) % 3 == 0, 0.15, 0.97)}[pattern].to(DEV)
    routed = (torch.rand(h_kv, n, T, device=DEV, generator=gen) < share[None, :, None]) & (chunk < own[:, None])
    bias = 0.5 * torch.randn(h_kv, n, T, device=DEV, generator=gen)
    out = B.alloc_routing(p)
    out["blk_bias"].zero_()
    start = torch.tensor([[B.dash_attn_list_offset(p, 0, r, i) for i in range(n)] for r in range(h_kv)], device=DEV)
    at = start[..., None] + routed.cumsum(2) - 1
    out["blk_bias"][at[routed]] = bias[routed]
    bits = torch.zeros(h_kv, n, words * 32, dtype=torch.bool, device=DEV)
    bits[:, :, :T] = routed
    bits[:, row, own] = True
    out["mask"][0] = (bits.view(h_kv, n, words, 32) * (2 ** torch.arange(32, device=DEV, dtype=torch.int64))).sum(3).to(torch.int32)
    return out, routed, bias, at


@pytest.mark.parametrize("pattern", ["few", "most", "all", "turns"])
@pytest.mark.parametrize("seq,h_q,h_kv,head_dim,block,one_term", [
    (1000, 2, 2, 64, 32, False), (1111, 2, 2, 128, 64, False), (450, 2, 2, 64, 16, False), (900, 4, 2, 128, 32, False), (1300, 8, 2, 64, 16, False),
    (1055, 8, 1, 64, 64, False), (777, 16, 1, 128, 16, False), (1200, 16, 1, 64, 128, False), (2100, 8, 2, 128, 64, True), (1030, 16, 1, 128, 128, True),
])
def test_runs_of_neighbours_against_float64(seq, h_q, h_kv, head_dim, block, one_term, pattern):
    gen = torch.Generator(DEV).manual_seed(81)
    rand = lambda h: torch.randn(1, seq, h, head_dim, device=DEV, generator=gen).bfloat16()
    Q, K, V, dO = rand(h_q), rand(h_kv), rand(h_kv), rand(h_q)
    p = B.params_for_prefill(Q, K, V, dO, block=block, alpha=1.5)
    rt, routed, bias, at = _routing(p, seq, h_kv, block, pattern, gen)
    dQ, dK = torch.empty_like(Q), torch.empty(1, seq, h_kv, head_dim, device=DEV)
    dV, db = torch.empty_like(dK), torch.empty_like(rt["blk_bias"])
    if one_term:
        ws = B.alloc_bwd_workspace(p)
        B.dash_attn_bwd_attend_prefill_tc(p, Q, K, V, dO, rt["mask"], rt["blk_bias"], dQ, dK, dV, db, ws)
        assert B.dash_attn_last_status(ws) == 0
    else:
        B.dash_attn_bwd_attend_prefill(p, Q, K, V, dO, rt["mask"], rt["blk_bias"], dQ, dK, dV, db)
    g, scale = h_q // h_kv, 1.0 / math.sqrt(head_dim)
    row, T = torch.arange(seq, device=DEV), routed.shape[2]
    own = row // block
    want = {k: torch.zeros(1, seq, h, head_dim, dtype=torch.double, device=DEV) for k, h in (("dQ", h_q), ("dK", h_kv), ("dV", h_kv))}
    want_b = torch.zeros(h_kv, seq, T, dtype=torch.double, device=DEV)
    for h in range(h_q):
        r = h // g
        b = torch.where(routed[r], bias[r].double(), -math.inf)
        b[row, own] = 0.0
        b = b[:, own].masked_fill(row[None] > row[:, None], -math.inf)
        q, k, v, do = Q[0, :, h].double(), K[0, :, r].double(), V[0, :, r].double(), dO[0, :, h].double()
        P = torch.softmax(q @ k.T * scale + b, -1)
        dP = do @ v.T
        dS = P * (dP - (P * dP).sum(-1, keepdim=True))
        want["dQ"][0, :, h] = dS @ k * scale
        want["dK"][0, :, r] += dS.T @ q * scale
        want["dV"][0, :, r] += P.T @ do
        want_b[r] += torch.zeros(seq, T, dtype=torch.double, device=DEV).index_add(1, own, dS)
    bound = 2.0 ** -8 if one_term else 2.0 ** -17
    for name, got, ref, rel in (("dQ", dQ, want["dQ"], 2.0 ** -8), ("dK", dK, want["dK"], bound), ("dV", dV, want["dV"], bound), ("dbias", db[at[routed]], want_b[routed], 8e-6)):
        err, norm = float((got.double() - ref).norm()), float(ref.norm())
        assert err <= rel * norm, (name, err / max(norm, 1e-300))
