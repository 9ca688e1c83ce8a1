"""Decode outputs carry no error beyond their own rounding to bf16: the weights enter the product with V as two bf16 terms
(2^-17 each), which disappears beside it.  The relative 2-norm error against the float64 oracle then is that of the rounded
oracle; one bf16 term per weight adds about 1.2e-3 in quadrature to 1.66e-3, a factor of 1.2."""
import numpy as np
import pytest
import torch

from oracle import dash_oracle as orc
from paper_2605_18753_b200 import binding as B
from paper_2605_18753_b200 import synth
from tests import helpers as H
from tests.test_gpu_parity import _wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch,seq,h_q,h_kv,head_dim,block", [
    (2, 2000, 8, 2, 128, 64), (3, 2000, 8, 4, 64, 16), (2, 3000, 32, 2, 128, 32),       # one launch, clusters
    (24, 1600, 16, 16, 64, 32), (20, 2500, 32, 16, 128, 64),                            # two kernels
    (24, 1400, 128, 8, 128, 128), (40, 900, 128, 8, 64, 16),                            # sixteen heads: a tile of their own
])
def test_decode_error_is_the_rounding_of_the_output(batch, seq, h_q, h_kv, head_dim, block):
    w = _wl(kind="decode", batch=batch, seq=seq, h_q=h_q, h_kv=h_kv, head_dim=head_dim, block=block, seed=81)
    inp = synth.make_decode_inputs(w, "cuda", kv_len=[seq - 97 * i % (seq // 2) for i in range(batch)])
    Q, K, V, lens = inp["Q"], inp["K"], inp["V"], inp["kv_len"]
    O = torch.empty_like(Q)
    p = B.params_for_decode(Q, K, V, O, block=block, alpha=w.alpha, gamma=w.gamma, sigma=w.sigma)
    kbar, ws = B.alloc_kbar(p), B.alloc_workspace(p)
    B.dash_attn_block_summaries(p, K, kbar, kv_len=lens)
    B.dash_attn_fwd_decode(p, Q, K, V, kbar, lens, O, ws)
    assert B.dash_attn_last_status(ws) == 0
    ref = orc.forward_decode(H.to_np64(Q), H.to_np64(K), H.to_np64(V), lens.cpu().numpy(), B=block, alpha=w.alpha, gamma=w.gamma, sigma=w.sigma)
    # a chunk on the threshold may fall to either side: groups that hold one are another function there
    keep = np.ones((batch, h_kv), dtype=bool)
    for (b, r), rt in ref["routing"].items():
        keep[b, r] = not (rt.n_cand and (np.abs(rt.margin) <= H.BORDERLINE).any())
    keep = np.repeat(keep, h_q // h_kv, axis=1)
    assert keep.sum() >= 8
    got, want = H.to_np64(O)[keep], ref["O"][keep]
    rounded = torch.from_numpy(want).to(torch.bfloat16).double().numpy()
    err, own = np.linalg.norm(got - want), np.linalg.norm(rounded - want)
    assert err <= 1.05 * own, (err / np.linalg.norm(want), own / np.linalg.norm(want))
