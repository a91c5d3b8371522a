"""Decode attention where heads are shared by warps and by CTAs in every way: fewer work units than CTAs, than warps, slices that
start and end inside a head, sequences of length 0 and 1 between long ones, and more sequences than a CTA plans by itself.
The workspace starts as garbage and the result is compared with the oracle's on the library's own cache."""
import numpy as np
import pytest

from paper_2609_38121_b200 import workloads as W
from tests.harness import Layer

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lengths,n_q,n_kv,bits,ctas", [
    ([70], 1, 1, 2, 148),                     # 9 units on 148 CTAs: every unit is another CTA's
    ([1, 900, 0, 333], 8, 2, 4, 200),         # an empty sequence, a one-token sequence, more CTAs than units of a head
    ([3000], 8, 1, 2, 31),                    # 56 units of one head over 31 CTAs of 12 warps: empty slices between the warps
    ([5000, 90], 3, 1, 2, 7),                 # slices of about one unit: a head across several CTAs
    ([200] * 150, 2, 1, 3, 3),                # many heads inside one warp's slice
    ([400] * 75, 14, 2, 2, 0),                # seven query heads, a CTA per SM or fewer
])
def test_shared_heads(lengths, n_q, n_kv, bits, ctas, test_option):
    import torch
    wl = W.LayerWorkload(dict(seed=83, batch=len(lengths), n_q=n_q, n_kv=n_kv, ctx=0, theta=1e4, bits=bits, s_sink=4, s_keep=64,
                              rmsnorm=False, ragged=None, prefill_chunk=0))
    L = Layer(wl, lengths, bits, 4, 64, 1, max_seq_len=max(lengths))
    L.fill()
    test_option("decode_ctas", ctas)
    B, dev = L.B, L.cache.device
    queries = np.stack([wl.queries(b, max(n - 1, 0)) for b, n in enumerate(lengths)])
    Q = torch.from_numpy(W.f32_to_bf16_bits(queries).view(np.int16)).to(dev)
    nbytes = B.decode_workspace_bytes(L.cache.desc, L.batch, L.max_seq_len)
    outs = []
    for _ in range(3):
        ws = torch.full((nbytes,), 0xFF, dtype=torch.uint8, device=dev)
        O = torch.full((L.batch, n_q, 128), float("nan"), device=dev)
        B.decode_attn(L.cache.desc, L.batch, L.slot, L.seq_len, L.max_seq_len, Q, O, ws, nbytes)
        torch.cuda.synchronize()
        outs.append(O.cpu().numpy())
    assert L.cache.status() == 0
    assert np.array_equal(outs[0], outs[1]) and np.array_equal(outs[0], outs[2])      # whichever CTA merges
    for b in sorted({0, len(lengths) // 2, len(lengths) - 1} | {b for b, n in enumerate(lengths) if n < 2}):
        if lengths[b] == 0:
            assert np.all(outs[0][b] == 0)
            continue
        ref = L.oracle_decode_on_gpu_cache(b, queries[b])
        assert np.max(np.abs(outs[0][b] - ref)) <= 2e-3 * np.max(np.abs(ref))


def test_more_sequences_than_a_cta_plans():
    """Above 8192 sequences the preparation kernel's first CTA writes the work plan, in the fused step behind the append that it waits
    for: the step and the two calls agree bit for bit, and with the oracle."""
    import torch
    n = 8500
    rng = np.random.default_rng(9)
    lengths = rng.integers(1, 90, n)
    lengths[[5, 4000, n - 1]] = 150
    wl = W.LayerWorkload(dict(seed=89, batch=n, n_q=2, n_kv=1, ctx=0, theta=1e4, bits=2, s_sink=4, s_keep=64, rmsnorm=False, ragged=None,
                              prefill_chunk=0))
    L = Layer(wl, lengths, 2, 4, 64, 1, max_seq_len=150)
    L.append_step(lengths - 1, oracle_too=False)
    B, dev = L.B, L.cache.device
    bits16 = lambda x: torch.from_numpy(W.f32_to_bf16_bits(x).view(np.int16)).to(dev)  # noqa: E731
    queries = W.bf16_round_f32(rng.standard_normal((n, 2, 128)).astype(np.float32))
    Q, K, V = bits16(queries), bits16(np.stack([L.tokens[b][0][-1] for b in range(n)])), bits16(np.stack([L.tokens[b][1][-1] for b in range(n)]))
    cu = torch.arange(n + 1, dtype=torch.int32, device=dev)
    nbytes = B.decode_workspace_bytes(L.cache.desc, n, 150)
    outs = [torch.full((n, 2, 128), float("nan"), device=dev) for _ in range(2)]
    ws = [torch.full((nbytes,), 0xFF, dtype=torch.uint8, device=dev) for _ in range(2)]
    B.decode_step(L.cache.desc, n, L.slot, L.seq_len, cu, 150, K, V, Q, outs[0], ws[0], nbytes)
    B.decode_attn(L.cache.desc, n, L.slot, L.seq_len, 150, Q, outs[1], ws[1], nbytes)
    torch.cuda.synchronize()
    assert L.cache.status() == 0
    assert np.array_equal(L.seq_len.cpu().numpy(), lengths)
    assert torch.equal(outs[0], outs[1])
    out = outs[0].cpu().numpy()
    assert np.all(np.isfinite(out))
    for b in [0, 5, 127, 128, 4000, 8191, 8192, n - 1]:
        ref = L.oracle_decode_on_gpu_cache(b, queries[b])
        assert np.max(np.abs(out[b] - ref)) <= 2e-3 * np.max(np.abs(ref))
