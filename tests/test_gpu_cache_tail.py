"""Cache rows behind kv_len may hold anything: a decode step must give the same bits whatever they are.  Lengths that leave a
block an odd and an even number of 64-token sub-blocks, own chunks of one token and full ones, every chunk size, the
one-launch step and the two kernels, contiguous and paged caches; and page-table entries behind the length, which are never
read, not even those that would follow the last entry of the table."""
import pytest
import torch

from paper_2605_18753_b200 import binding as B
from paper_2605_18753_b200 import synth
from tests.test_gpu_paged import _scatter_into_pages
from tests.test_gpu_parity import _wl

pytestmark = pytest.mark.gpu
DEV = "cuda"


def _decode(w, Q, K, V, lens, page_size):
    O = torch.full_like(Q, float("nan"))
    opt = dict(block=w.block, alpha=w.alpha, gamma=w.gamma, sigma=w.sigma)
    if page_size:
        Kp, Vp, table = _scatter_into_pages(K, V, page_size, seed=3)
        p = B.params_for_paged_decode(Q, Kp, Vp, O, max_pages=table.shape[1], **opt)
        kbar, ws = B.alloc_kbar(p).zero_(), B.alloc_workspace(p)
        B.dash_attn_block_summaries_paged(p, Kp, table, kbar, kv_len=lens)
        B.dash_attn_fwd_decode_paged(p, Q, Kp, Vp, table, kbar, lens, O, ws)
    else:
        p = B.params_for_decode(Q, K, V, O, **opt)
        kbar, ws = B.alloc_kbar(p).zero_(), B.alloc_workspace(p)
        B.dash_attn_block_summaries(p, K, kbar, kv_len=lens)
        B.dash_attn_fwd_decode(p, Q, K, V, kbar, lens, O, ws)
    assert B.dash_attn_last_status(ws) == 0
    return O


@pytest.mark.parametrize("block", [16, 32, 64, 128])
@pytest.mark.parametrize("batch,h_kv,g_q,head_dim,page_size", [
    (12, 1, 4, 128, 0), (30, 2, 2, 64, 0), (12, 2, 16, 64, 0),            # one launch: clusters of 8, 4 and 8
    (50, 4, 4, 128, 0), (40, 8, 1, 64, 0),                                # two kernels, in one wave and in several
    (12, 1, 8, 64, 256), (50, 4, 2, 128, 128),                            # paged
])
def test_rows_behind_the_length_do_not_matter(block, batch, h_kv, g_q, head_dim, page_size):
    w = _wl(kind="decode", batch=batch, seq=1536, h_q=g_q * h_kv, h_kv=h_kv, head_dim=head_dim, block=block, seed=90 + block)
    # own chunks of 1, B - 1, B and a few other tokens, after 0, 1, 2, ... complete chunks
    lens = [max(1, min(1536, (i * 7 % (1536 // block)) * block + (1, block - 1, block, block // 2 + 1)[i % 4])) for i in range(batch)]
    inp = synth.make_decode_inputs(w, DEV, kv_len=lens)
    Q, K, V, kv = inp["Q"], inp["K"], inp["V"], inp["kv_len"]
    behind = (torch.arange(1536, device=DEV)[None] >= kv[:, None])[..., None, None]
    outs = []
    for fill in (0.0, float("nan"), float("inf")):
        outs.append(_decode(w, Q, K.masked_fill(behind, fill), V.masked_fill(behind, fill), kv, page_size))
    assert torch.isfinite(outs[0].float()).all()
    assert torch.equal(outs[0], outs[1]) and torch.equal(outs[0], outs[2])


@pytest.mark.parametrize("block", [16, 32, 64, 128])
@pytest.mark.parametrize("batch,h_kv,page_size", [(12, 1, 128), (50, 4, 128), (12, 2, 256)])
def test_table_entries_behind_the_length_are_not_read(block, batch, h_kv, page_size):
    """The debug library reports every page id outside the pool that a kernel reads; the table sits at the end of its buffer,
    with such ids right behind it."""
    w = _wl(kind="decode", batch=batch, seq=1536, h_q=2 * h_kv, h_kv=h_kv, head_dim=64, block=block, seed=95 + block)
    per = 1536 // page_size
    # lengths that end in the last chunk of a page, the whole table's last page included, and in other chunks
    lens = [(i % per + 1) * page_size - (0, 1, block - 1, block, 3 * block)[i % 5] % page_size for i in range(batch - 1)] + [1536]
    inp = synth.make_decode_inputs(w, DEV, kv_len=lens)
    Q, K, V, kv = inp["Q"], inp["K"], inp["V"], inp["kv_len"]
    want = _decode(w, Q, K, V, kv, 0)
    Kp, Vp, table = _scatter_into_pages(K, V, page_size, seed=4)
    used = -(-kv // page_size)
    for bad in (-1, Kp.shape[0] + 5):
        buffer = torch.full((batch * per + 64,), bad, dtype=torch.int32, device=DEV)
        t = buffer[:batch * per].view(batch, per)
        t.copy_(table.masked_fill(torch.arange(per, device=DEV)[None] >= used[:, None], bad))
        O = torch.full_like(Q, float("nan"))
        p = B.params_for_paged_decode(Q, Kp, Vp, O, max_pages=per, block=block, alpha=w.alpha, gamma=w.gamma, sigma=w.sigma)
        with B.use_debug_library():
            kbar, ws = B.alloc_kbar(p).zero_(), B.alloc_workspace(p)
            B.dash_attn_block_summaries_paged(p, Kp, t, kbar, kv_len=kv)
            B.dash_attn_fwd_decode_paged(p, Q, Kp, Vp, t, kbar, kv, O, ws)
            assert B.dash_attn_last_status(ws) == 0
        assert torch.equal(O, want)
