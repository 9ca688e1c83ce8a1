"""Expanded tensors (stride 0 over the batch or over the KV heads): every entry point must give what it gives for the same
values written out.  The written-out call may take other kernels, so the comparison carries the tolerances of the dtype."""
import pytest
import torch

from paper_2605_18753_b200 import binding as B
from tests import helpers as H

pytestmark = pytest.mark.gpu
DEV = "cuda"


def _rand(seed, *shape):
    return torch.randn(*shape, device=DEV, generator=torch.Generator(DEV).manual_seed(seed)).to(torch.bfloat16)


def _same(got, want, what, rel=None):
    if rel is None:
        H.check_outputs(H.to_np64(got), H.to_np64(want), torch.bfloat16, what)
    else:
        scale = max(1.0, float(want.abs().max()))
        assert float((got.double() - want.double()).abs().max()) <= rel * scale, what


@pytest.mark.parametrize("g_q,block", [(1, 32), (1, 64), (4, 64)])
@pytest.mark.parametrize("what", ["kv heads", "kv batch", "q batch"])
def test_prefill_and_backward(g_q, block, what):
    b, n, h_kv, d = 2, 500, 4, 64
    h_q = g_q * h_kv
    Q, K, V, dO = _rand(1, b, n, h_q, d), _rand(2, b, n, h_kv, d), _rand(3, b, n, h_kv, d), _rand(4, b, n, h_q, d)
    if what == "kv heads":
        K, V = K[:, :, :1].expand(b, n, h_kv, d), V[:, :, :1].expand(b, n, h_kv, d)
    elif what == "kv batch":
        K, V = K[:1].expand(b, n, h_kv, d), V[:1].expand(b, n, h_kv, d)
    else:
        Q = Q[:1].expand(b, n, h_q, d)
    opt = dict(block=block, alpha=1.5, gamma=2.0, sigma=2.0)
    outs = []
    for q, k, v in ((Q, K, V), (Q.contiguous(), K.contiguous(), V.contiguous())):
        O = torch.full((b, n, h_q, d), float("nan"), device=DEV, dtype=torch.bfloat16)
        p = B.params_for_prefill(q, k, v, O, **opt)
        ws = B.alloc_workspace(p)
        B.dash_attn_fwd_prefill(p, q, k, v, O, ws)
        assert B.dash_attn_last_status(ws) == 0
        kbar, rt = B.alloc_kbar(p), B.alloc_routing(p, with_tau=True)
        for t in rt.values():
            t.zero_()
        B.dash_attn_block_summaries(p, k, kbar)
        B.dash_attn_select(p, q, kbar, rt["mask"], rt["count"], rt["blk_idx"], rt["blk_bias"], ws, tau=rt["tau"])
        outs.append((O, rt))
    (O0, rt0), (O1, rt1) = outs
    # (a chunk on the threshold may fall to either side of it on different kernels)
    same = (rt0["mask"] == rt1["mask"]).all(-1).permute(0, 2, 1).repeat_interleave(g_q, dim=2)
    assert same.float().mean() > 0.97 and torch.allclose(rt0["tau"], rt1["tau"], rtol=0, atol=2e-5)
    _same(O0[same], O1[same], "fwd_prefill")
    # backward on one routing
    if what != "q batch":                 # (dQ has the strides of Q)
        grads = []
        for k, v in ((K, V), (K.contiguous(), V.contiguous())):
            p = B.params_for_prefill(Q, k, v, dO, **opt)
            dQ, dK = torch.empty_like(Q), torch.empty(b, n, h_kv, d, device=DEV)
            dV, db = torch.empty_like(dK), torch.empty_like(rt1["blk_bias"])
            B.dash_attn_bwd_attend_prefill(p, Q, k, v, dO, rt1["mask"], rt1["blk_bias"], dQ, dK, dV, db)
            grads.append((dQ, dK, dV, db))
        for x, y, name in zip(*grads, ("dQ", "dK", "dV", "dbias")):
            _same(x, y, name, 1e-2 if name == "dQ" else 2e-4)


def test_backward_of_an_expanded_gradient():
    b, n, h_q, h_kv, d = 2, 300, 4, 4, 64
    Q, K, V = _rand(5, b, n, h_q, d), _rand(6, b, n, h_kv, d), _rand(7, b, n, h_kv, d)
    dO = _rand(8, 1, 1, h_q, d).expand(b, n, h_q, d)        # as the gradient of a sum over tokens arrives
    opt = dict(block=32, alpha=1.5, gamma=2.0, sigma=2.0)
    p = B.params_for_prefill(Q, K, V, Q, **opt)
    ws, kbar, rt = B.alloc_workspace(p), B.alloc_kbar(p), B.alloc_routing(p)
    B.dash_attn_block_summaries(p, K, kbar)
    B.dash_attn_select(p, Q, kbar, rt["mask"], rt["count"], rt["blk_idx"], rt["blk_bias"], ws)
    grads = []
    for g in (dO, dO.contiguous()):
        p = B.params_for_prefill(Q, K, V, g, **opt)
        dQ, dK = torch.empty_like(Q), torch.empty(b, n, h_kv, d, device=DEV)
        dV, db = torch.empty_like(dK), torch.zeros_like(rt["blk_bias"])
        B.dash_attn_bwd_attend_prefill(p, Q, K, V, g, rt["mask"], rt["blk_bias"], dQ, dK, dV, db)
        grads.append((dQ, dK, dV, db))
    for x, y, name in zip(*grads, ("dQ", "dK", "dV", "dbias")):
        _same(x, y, name, 1e-2 if name == "dQ" else 2e-4)


@pytest.mark.parametrize("g_q,batch", [(1, 2), (4, 2), (4, 60)])      # one launch and two kernels, where written out
@pytest.mark.parametrize("what", ["kv heads", "kv batch"])
def test_decode(g_q, batch, what):
    n, h_kv, d = 900, 4, 128
    Q, K, V = _rand(11, batch, g_q * h_kv, d), _rand(12, batch, n, h_kv, d), _rand(13, batch, n, h_kv, d)
    if what == "kv heads":
        K, V = K[:, :, :1].expand(batch, n, h_kv, d), V[:, :, :1].expand(batch, n, h_kv, d)
    else:
        K, V = K[:1].expand(batch, n, h_kv, d), V[:1].expand(batch, n, h_kv, d)
    lens = torch.tensor([n - 13 * (i % 50) for i in range(batch)], dtype=torch.int32, device=DEV)
    outs = []
    for k, v in ((K, V), (K.contiguous(), V.contiguous())):
        O = torch.full_like(Q, float("nan"))
        p = B.params_for_decode(Q, k, v, O, block=32, alpha=1.5, gamma=0.1, sigma=2.0)      # (small logits: no chunk near the threshold)
        kbar, ws = B.alloc_kbar(p), B.alloc_workspace(p)
        B.dash_attn_block_summaries(p, k, kbar, kv_len=lens)
        B.dash_attn_fwd_decode(p, Q, k, v, kbar, lens, O, ws)
        assert B.dash_attn_last_status(ws) == 0
        outs.append(O)
    _same(outs[0], outs[1], "fwd_decode")
