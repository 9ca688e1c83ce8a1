"""Stage-2 backward on tensor cores at the edges of its tiles: query tiles over several chunks, key slices that hold one
chunk or several, both head dims, sequence ends at slice, tile and chunk edges, and slices whose query tiles are shared by
several blocks.  Against the float64 oracle with the tolerances of the entry point's fp32 gradients."""
import pytest

from tests.test_gpu_backward import test_stage2_backward_matches_oracle as against_oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("g_q,block", [(1, 16), (1, 64), (1, 128), (2, 16), (2, 32), (2, 128), (4, 16), (4, 32), (16, 64)])
@pytest.mark.parametrize("head_dim,seq,local_blocks", [(64, 257, 0), (128, 319, 1)])
def test_backward_tiles(g_q, block, head_dim, seq, local_blocks):
    against_oracle(dict(seq=seq, h_q=2 * g_q, h_kv=2, head_dim=head_dim, block=block, gamma=2.0, seed=60 + g_q), local_blocks)
