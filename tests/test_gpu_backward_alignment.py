"""The fp32 buffers of the routing and summary backward calls may sit anywhere a float may, as views into a flat gradient buffer
do: every offset must give what 16-byte aligned buffers give (up to the order of the atomic sums)."""
import pytest
import torch

from paper_2605_18753_b200 import binding as B
from paper_2605_18753_b200 import synth
from tests.test_gpu_parity import _wl

pytestmark = pytest.mark.gpu
DEV = "cuda"


def _at(t, offset):
    """The same values `offset` floats behind a 16-byte boundary."""
    flat = torch.full((t.numel() + 8,), float("nan"), device=DEV)
    view = flat[offset:offset + t.numel()].view(t.shape)
    view.copy_(t)
    return view


@pytest.mark.parametrize("dtype,h_q,head_dim", [("bf16", 4, 64), ("bf16", 32, 128), ("f32", 2, 128), ("f32", 8, 64)])
@pytest.mark.parametrize("offset", [1, 2, 3])
def test_offset_buffers(dtype, h_q, head_dim, offset):
    w = _wl(seq=300, h_q=h_q, h_kv=2, head_dim=head_dim, block=16, dtype=dtype, gamma=2.0, seed=61)
    inp = synth.make_prefill_inputs(w, DEV)
    Q, K = inp["Q"], inp["K"]
    p = B.params_for_prefill(Q, K, inp["V"], Q, block=16, alpha=w.alpha, gamma=w.gamma, sigma=w.sigma)
    g = torch.Generator(DEV).manual_seed(62)
    qbar = torch.randn(2, head_dim, generator=g, device=DEV)
    kbar, ws, rt = B.alloc_kbar(p), B.alloc_workspace(p), B.alloc_routing(p, with_tau=True)
    B.dash_attn_block_summaries(p, K, kbar, qbar)
    B.dash_attn_select(p, Q, kbar, rt["mask"], rt["count"], rt["blk_idx"], rt["blk_bias"], ws, tau=rt["tau"])
    dbias = torch.randn(rt["blk_bias"].shape, generator=g, device=DEV)
    dK = torch.randn(w.batch, w.seq, 2, head_dim, generator=g, device=DEV)

    def run(place):
        dQr, dKbar = place(torch.zeros(Q.shape, device=DEV)), place(torch.zeros_like(kbar))
        B.dash_attn_bwd_select_prefill(p, Q, place(kbar), rt["count"], rt["blk_idx"], rt["tau"], dbias, dQr, dKbar)
        out, dqbar = place(dK), place(torch.zeros_like(qbar))
        B.dash_attn_bwd_block_summaries(p, K, place(dKbar), out, place(qbar), 0, dqbar)
        return dQr, dKbar, out, dqbar

    want = run(lambda t: t.clone())
    for got, ref, name in zip(run(lambda t: _at(t, offset)), want, ("dQ_route", "dKbar", "dK", "dqbar")):
        # sums of up to 300 * 16 products in fp32, in another order: 2^-24 each, of the largest value
        assert torch.isfinite(got).all() and float((got - ref).abs().max()) <= 1e-4 * float(ref.abs().max()), name
