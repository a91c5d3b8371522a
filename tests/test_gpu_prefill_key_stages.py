"""Key stages of the chunk attention kernel where they pass from the staging threads to bulk tensor copies and back to free: chunk tiles that
begin at an even or odd place of a CTA's key tiles, a last tile that only one of the two query tiles sees, staged tiles ahead of
them (none, window rows, packed pages with ends outside the quantized range), whole or cut into shares, against the oracle's
chunk_attn."""
import pytest

from paper_2609_38121_b200 import workloads as W
from tests.harness import Layer

pytestmark = pytest.mark.gpu

CONTEXTS = [1, 40, 64, 100, 230, 300]
CHUNKS = [65, 129, 200, 64, 321, 190]


@pytest.mark.parametrize("copies", [True, False])
@pytest.mark.parametrize("bits,n_q,turn,split", [(2, 8, 0, 1), (2, 8, 2, 2), (3, 8, 1, 1), (3, 14, 4, 3), (4, 8, 3, 5), (4, 2, 5, 1)])
def test_stages_from_staging_threads_to_copies(bits, n_q, turn, split, copies, test_option):
    test_option("prefill_split", split)
    if not copies:
        test_option("prefill_no_tma", 1)
    wl = W.LayerWorkload(dict(seed=101, batch=len(CONTEXTS), n_q=n_q, n_kv=2, ctx=0, theta=1e4, bits=bits, s_sink=4, s_keep=64,
                              rmsnorm=False, ragged=None, prefill_chunk=0))
    counts = CHUNKS[turn:] + CHUNKS[:turn]
    L = Layer(wl, [c + n for c, n in zip(CONTEXTS, counts)], bits, 4, 64, 8, page_shuffle_seed=3)
    L.append_step(CONTEXTS)
    assert L.check_prefill_parity(counts) <= 2e-3
    assert L.cache.status() == 0


@pytest.mark.parametrize("n", [127, 128, 130, 192, 256, 511])
def test_prompt_lengths_around_tiles(n, test_option):
    """A prompt alone, uncut: the chunk's tiles are the only ones; the second query tile sees up to one key tile more than the first."""
    test_option("prefill_split", 1)
    wl = W.LayerWorkload(dict(seed=102, batch=1, n_q=4, n_kv=1, ctx=0, theta=1e4, bits=2, s_sink=4, s_keep=64, rmsnorm=False, ragged=None,
                              prefill_chunk=0))
    L = Layer(wl, [n], 2, 4, 64, 1)
    assert L.check_prefill_parity([n]) <= 2e-3
    assert L.cache.status() == 0


@pytest.mark.parametrize("n,ctx,split", [(522, 0, 1), (522, 300, 1), (538, 300, 2), (1030, 0, 3)])
def test_last_pair_without_a_second_tile(n, ctx, split, test_option):
    """Four heads per key/value head: a query tile is 32 positions, a pair 64.  The last pair has positions for its first tile only, and more
    copied key tiles than stages, which the second tile's issuing warp passes over."""
    test_option("prefill_split", split)
    wl = W.LayerWorkload(dict(seed=103, batch=1, n_q=8, n_kv=2, ctx=0, theta=1e4, bits=2, s_sink=4, s_keep=64, rmsnorm=False, ragged=None,
                              prefill_chunk=0))
    L = Layer(wl, [ctx + n], 2, 4, 64, 1)
    if ctx:
        L.append_step([ctx])
    assert L.check_prefill_parity([n]) <= 2e-3
    assert L.cache.status() == 0
