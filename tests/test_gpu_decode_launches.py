"""Decode steps on both sides of every line between their launches: clusters of 8, 4 and 2 blocks per (batch, KV head) and the
two kernels behind them, caches of 512 and 513 chunks, shares of a list that leave blocks without work, and grids of several
waves in which short lists take fewer splits than the grid has.  Against the oracle."""
import pytest

from tests import test_gpu_parity as P

pytestmark = pytest.mark.gpu


def _lens(seq, batch):
    return [seq] + [1 + (i * 37) % seq for i in range(1, batch)]


@pytest.mark.parametrize("batch,h_kv", [(1, 1), (37, 1), (19, 2), (37, 2), (25, 3), (74, 2), (75, 2), (150, 2)])
def test_cluster_sizes_and_waves(batch, h_kv):
    w = P._wl(kind="decode", batch=batch, seq=400, h_q=4 * h_kv, h_kv=h_kv, head_dim=64, block=32, gamma=2.0, seed=70)
    P._decode_case(w, _lens(400, batch))


@pytest.mark.parametrize("chunks", [512, 513])
# (sixteen heads: one KV head and three sequences, because from 64 rows on the harness wants four fifths of the groups free of
# chunks inside the 1e-4 band around the threshold, which so many heads seldom are)
@pytest.mark.parametrize("g_q,head_dim,h_kv,batch", [(1, 128, 2, 2), (8, 64, 2, 2), (16, 64, 1, 3), (16, 128, 1, 3)])
def test_longest_fused_cache(chunks, g_q, head_dim, h_kv, batch):
    w = P._wl(kind="decode", batch=batch, seq=chunks * 16 + 5, h_q=h_kv * g_q, h_kv=h_kv, head_dim=head_dim, block=16, seed=71)
    P._decode_case(w, [chunks * 16 + 5, 700, chunks * 8][:batch], local_blocks=1)
