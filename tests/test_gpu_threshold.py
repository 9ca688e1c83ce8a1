"""Thresholds of the routing where the iteration ends on a step instead of a pass that confirms it: every row's threshold against
the exact root over float64 logits, for exponents 2 and 4 (which have the rule) and 1 (which has not), rows of up to 8, 128,
256, 512 and more candidates.

The iteration stops at |F - 1| <= 4e-6 or after a step that leaves at most that; |dF / dtau| >= 1 at the root, and the logits carry
fp32-class sums (2e-6 of the largest): 8e-6 of max(1, |x|) covers both."""
import math

import pytest
import torch

from paper_2605_18753_b200 import binding as B
from paper_2605_18753_b200 import synth
from tests.test_gpu_parity import _wl

pytestmark = pytest.mark.gpu
DEV = "cuda"


def _root(x, e):
    """The root of sum [x - tau]_+^e = 1 over the last dimension (-inf: no candidate)."""
    hi = x.amax(-1)
    lo = hi - 1.0
    for _ in range(60):
        mid = 0.5 * (lo + hi)
        above = (x - mid[..., None]).clamp(min=0.0).pow(e).sum(-1) >= 1.0
        lo, hi = torch.where(above, mid, lo), torch.where(above, hi, mid)
    return 0.5 * (lo + hi)


@pytest.mark.parametrize("alpha", [1.25, 1.5, 2.0])
@pytest.mark.parametrize("seq,block,h_q,h_kv", [(300, 32, 8, 2), (4200, 32, 4, 1), (4100, 16, 4, 1), (8300, 16, 4, 2), (17000, 16, 8, 1), (2000, 16, 2, 2)])
def test_prefill_thresholds_are_the_root(alpha, seq, block, h_q, h_kv):
    w = _wl(seq=seq, h_q=h_q, h_kv=h_kv, head_dim=64, block=block, alpha=alpha, seed=91)
    inp = synth.make_prefill_inputs(w, DEV)
    Q, K = inp["Q"], inp["K"]
    p = B.params_for_prefill(Q, K, inp["V"], Q, block=block, alpha=alpha, gamma=w.gamma, sigma=w.sigma)
    ws, kbar, rt = B.alloc_workspace(p), B.alloc_kbar(p), B.alloc_routing(p, with_tau=True)
    B.dash_attn_block_summaries(p, K, kbar)
    B.dash_attn_select(p, Q, kbar, rt["mask"], rt["count"], rt["blk_idx"], rt["blk_bias"], ws, tau=rt["tau"])
    assert B.dash_attn_last_status(ws) == 0
    rows = torch.cat([torch.arange(block, min(seq, 8 * block)), torch.linspace(block, seq - 1, 257).long()]).unique().to(DEV)
    cand = torch.arange(seq // block, device=DEV)[None] < (rows // block)[:, None]
    for h in range(h_q):
        x = Q[0, rows, h].double() @ kbar[0, h // (h_q // h_kv)].double().T * (w.gamma * (alpha - 1.0) / math.sqrt(64))
        x = x.masked_fill(~cand, -math.inf)
        want, got = _root(x, 1.0 / (alpha - 1.0)), rt["tau"][0, h, rows].double()
        bound = 8e-6 * x.masked_fill(~cand, 0.0).abs().amax(-1).clamp(min=1.0)
        assert ((got - want).abs() <= bound).all(), float(((got - want).abs() / bound).max())
