"""Many short chunks on the tensor-core append path (its tiles then mix sequences): ragged counts, sequences without new tokens, a
token count that is no multiple of the tile, projected keys, transforms that are not bf16-valued; codes, scales and offsets against
the oracle's."""
import numpy as np
import pytest

from paper_2609_38121_b200 import workloads as W
from tests.harness import CODE_MISMATCH_MAX, Layer
from tests.test_gpu_projected import _compare_caches, _pair, _wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bits", [2, 3, 4])
def test_many_short_chunks(bits):
    n = 20                                              # about 45 new tokens each, 8 heads: over one token per warp of the rows path
    wl = W.LayerWorkload(dict(seed=141, batch=n, n_q=8, n_kv=8, ctx=0, theta=1e4, bits=bits, s_sink=4, s_keep=64, rmsnorm=False, ragged=None,
                              prefill_chunk=0))
    rng = np.random.default_rng(3)
    first, more = rng.integers(1, 70, n), rng.integers(30, 100, n)
    more[[2, 9]] = 0
    L = Layer(wl, first + more, bits, 4, 64, 1)
    L.append_step(first)
    L.append_step(more)
    assert L.cache.status() == 0
    assert L.check_append_parity() <= CODE_MISMATCH_MAX
    assert np.array_equal(L.seq_len.cpu().numpy(), first + more)


@pytest.mark.parametrize("bits,normalise,weights", [(2, True, True), (4, True, False), (3, False, False)])
def test_many_short_projected_chunks(bits, normalise, weights):
    """Every token of a tile is normalised and rotated for its own sequence's position, in tiles that mix sequences of different
    lengths, with sequences that bring nothing between them: against the same keys prepared by the oracle."""
    wl = _wl(47, 24, 8, 8, bits, theta=1e4)
    rng = np.random.default_rng(5)
    first, more = rng.integers(1, 70, 24), rng.integers(30, 100, 24)
    more[[0, 7, 8, 23]] = 0
    assert sum(first) > 592 and sum(more) > 592         # 17 tokens and more per CTA of the rows path: three per warp
    plain, fused, masks, _ = _pair(wl, first + more, bits, normalise, weights)
    for L in (plain, fused):
        L.append_step(first)
        L.append_step(more)
        assert L.cache.status() == 0
    assert plain.check_append_parity() <= CODE_MISMATCH_MAX
    share, rate = _compare_caches(plain, fused, masks, first + more, wl.n_kv)
    assert share <= 0.25 and rate <= 0.05


@pytest.mark.parametrize("bits,n", [(2, 20), (4, 60)])
def test_transforms_of_full_precision(bits, n):
    """A T_K whose entries are no bf16 values (the library's own are): short chunks are transformed by it as it is (several
    tiles per CTA: test_full_precision_over_several_tiles)."""
    from oracle import wushkv_oracle as O
    import torch
    wl = W.LayerWorkload(dict(seed=151, batch=n, n_q=8, n_kv=8, ctx=0, theta=1e4, bits=bits, s_sink=4, s_keep=64, rmsnorm=False, ragged=None,
                              prefill_chunk=0))
    new = np.random.default_rng(4).integers(30, 100, n)
    L = Layer(wl, new, bits, 4, 64, 1)
    T = (np.asarray(L.T) * 1.003).astype(np.float32)
    assert np.any(T != W.bf16_round_f32(T))
    L.cache.T_K.copy_(torch.from_numpy(T))
    L.oracle = [O.LayerCache(wl.n_kv, 128, bits, L.kappa_k, L.kappa_v, T.astype(np.float64)) for _ in range(n)]
    L.append_step(new)
    assert L.cache.status() == 0
    assert L.check_append_parity() <= CODE_MISMATCH_MAX


def test_full_precision_over_several_tiles():
    """64 heads leave four CTAs per head: each multiplies several tiles and puts the first term of T_K back between them."""
    from oracle import wushkv_oracle as O
    import torch
    wl = W.LayerWorkload(dict(seed=153, batch=12, n_q=64, n_kv=64, ctx=0, theta=1e4, bits=2, s_sink=4, s_keep=64, rmsnorm=False, ragged=None,
                              prefill_chunk=0))
    new = np.full(12, 110)                              # 1320 tokens: 11 tiles
    L = Layer(wl, new, 2, 4, 64, 1)
    T = (np.asarray(L.T) * 1.003).astype(np.float32)
    L.cache.T_K.copy_(torch.from_numpy(T))
    L.oracle = [O.LayerCache(wl.n_kv, 128, 2, L.kappa_k, L.kappa_v, T.astype(np.float64)) for _ in range(12)]
    L.append_step(new)
    assert L.cache.status() == 0
    assert L.check_append_parity() <= CODE_MISMATCH_MAX
