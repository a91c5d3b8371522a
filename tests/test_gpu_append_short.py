"""Many short chunks on the tensor-core append path (its tiles then mix sequences): ragged counts, sequences without new tokens, a
token count that is no multiple of the tile, projected keys; codes, scales and offsets against the oracle's."""
import numpy as np
import pytest

from paper_2609_38121_b200 import workloads as W
from tests.harness import CODE_MISMATCH_MAX, Layer

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bits,projected", [(2, False), (3, False), (4, True)])
def test_many_short_chunks(bits, projected):
    n = 20                                              # about 45 new tokens each, 8 heads: over two (three) tokens per warp
    wl = W.LayerWorkload(dict(seed=141, batch=n, n_q=8, n_kv=8, ctx=0, theta=1e4, bits=bits, s_sink=4, s_keep=64, rmsnorm=False, ragged=None,
                              prefill_chunk=0))
    rng = np.random.default_rng(3)
    first, more = rng.integers(1, 70, n), rng.integers(30, 100, n)
    more[[2, 9]] = 0
    L = Layer(wl, first + more, bits, 4, 64, 1)
    if projected:                                       # keys as given, rotated by the angle 0 of a table whose base is huge
        from paper_2609_38121_b200 import binding as B
        L.prologue = B.Prologue(1e300, 1)
        L.prologue.table[..., 0], L.prologue.table[..., 1] = 1.0, 0.0
    L.append_step(first)
    L.append_step(more)
    if projected:
        assert L.cache.status() & ~L.B.DEV_ROPE_RANGE == 0
    else:
        assert L.cache.status() == 0
    assert L.check_append_parity() <= CODE_MISMATCH_MAX
    assert np.array_equal(L.seq_len.cpu().numpy(), first + more)
