"""Query tiles that span several chunks (chunks shorter than 128 / g_q tokens, and every chunk size with one query head
per KV head): sequence lengths at the edges of chunks, tiles and tile pairs, with and without the window, against the
oracle; every row of a tile has its own causal chunk, its own candidates and its own list."""
import pytest

from tests import test_gpu_parity as P

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("g_q,block", [(1, 16), (1, 32), (1, 64), (1, 128), (2, 16), (2, 32), (4, 16)])
@pytest.mark.parametrize("extra,local_blocks", [(-1, 0), (1, 1), (17, 2)])
def test_tiles_over_several_chunks(g_q, block, extra, local_blocks):
    tile = 128 // g_q
    for tiles, head_dim in ((1, 64), (5, 128)):
        seq = tiles * max(tile, block) + extra
        w = P._wl(seq=seq, h_q=2 * g_q, h_kv=2, head_dim=head_dim, block=block, dtype="bf16", gamma=2.0, seed=40 + tiles)
        P._fwd_prefill_case(w, range(seq), local_blocks=local_blocks)
