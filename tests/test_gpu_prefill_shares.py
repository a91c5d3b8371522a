"""Chunk attention whose tile pairs are shared by several CTAs by the amount of work: ragged chunks on ragged contexts, sequences
without new tokens, one long sequence among short ones, one key tile per share, and a workspace that holds fewer shares than
the call would like.  Against the oracle on the library's own cache, with the repository's tolerance."""
import numpy as np
import pytest

from paper_2609_38121_b200 import workloads as W
from tests.harness import Layer

pytestmark = pytest.mark.gpu


def _wl(n_q, n_kv, batch):
    return W.LayerWorkload(dict(seed=131, batch=batch, n_q=n_q, n_kv=n_kv, ctx=0, theta=1e4, bits=2, s_sink=4, s_keep=64, rmsnorm=False,
                                ragged=None, prefill_chunk=0))


@pytest.mark.parametrize("ctx,new,n_q,n_kv,bits", [
    ([2500], [3], 8, 1, 2),                                     # one pair, many shares
    ([0], [300], 8, 2, 2),                                      # no context: shares of one tile, causal pairs of different length
    ([1800, 40, 0, 700], [5, 90, 17, 0], 8, 2, 3),              # one long among short, a sequence without new tokens
    ([100] * 9 + [1500], [40] * 9 + [70], 14, 2, 4),            # one sequence worth several of the others
])
def test_shares_by_amount_of_work(ctx, new, n_q, n_kv, bits):
    L = Layer(_wl(n_q, n_kv, len(ctx)), [c + n for c, n in zip(ctx, new)], bits, 4, 64, 1)
    if sum(ctx):
        L.append_step(ctx)
    assert L.check_prefill_parity(new) <= 2e-3
    assert L.cache.status() == 0


def test_more_sequences_than_the_table_takes_at_once():
    """Above 512 sequences the table of shares is put together in two trips, and with more shares than SMs the pairs are sorted by the
    size of their shares: 560 short chunks on uneven contexts."""
    rng = np.random.default_rng(7)
    ctx, new = rng.integers(0, 200, 560), rng.integers(1, 6, 560)
    ctx[[3, 300, 530]] = [2000, 900, 1500]
    new[[10, 511, 512]] = 0
    L = Layer(_wl(8, 1, 560), ctx + new, 2, 4, 64, 1)
    L.append_step(ctx)
    assert L.check_prefill_parity(new) <= 2e-3
    assert L.cache.status() == 0


def test_smaller_workspaces():
    import torch
    from paper_2609_38121_b200 import binding as B
    ctx, new = [1200, 300], [20, 40]
    L = Layer(_wl(8, 2, 2), [c + n for c, n in zip(ctx, new)], 2, 4, 64, 1)
    L.append_step(ctx)
    L.prefill(new)
    full, total = L.first, sum(new)
    bits16 = lambda x: torch.from_numpy(W.f32_to_bf16_bits(x).view(np.int16)).cuda()  # noqa: E731
    K = bits16(np.concatenate([L.tokens[b][0][ctx[b]:ctx[b] + new[b]] for b in range(2)]))
    V = bits16(np.concatenate([L.tokens[b][1][ctx[b]:ctx[b] + new[b]] for b in range(2)]))
    Q = bits16(np.concatenate([L.wl.chunk_queries(b, np.arange(ctx[b], ctx[b] + new[b])) for b in range(2)]))
    cu = torch.tensor([0, 20, 60], dtype=torch.int32, device="cuda")
    # The least that is accepted: operands, then 16 shares of 528-byte rows (60 tokens x 8 heads; 2 CTAs without shares on the GPU).
    up = lambda x: (x + 255) // 256 * 256  # noqa: E731
    operands = 2 * up(total * 2 * 256) + up(2 * total * 8 * 256) + up(total * 8 * 4)
    least = up(operands + 16 * total * 8 * 528)
    asked = B.prefill_workspace_bytes(L.cache.desc, 2, total)
    assert asked >= least
    for nbytes in (asked, asked - 1, least):
        ws = torch.full((nbytes,), 0xFF, dtype=torch.uint8, device="cuda")
        O = torch.full((total, 8, 128), float("nan"), device="cuda")
        B.prefill_attn(L.cache.desc, 2, L.slot, L.seq_len, cu, total, 40, K, V, Q, O, ws, nbytes)
        torch.cuda.synchronize()
        assert np.max(np.abs(O.cpu().numpy() - full)) <= 1e-3 * np.max(np.abs(full))
    with pytest.raises(B.WushkvError) as e:
        B.prefill_attn(L.cache.desc, 2, L.slot, L.seq_len, cu, total, 40, K, V, Q, O, ws, least - 1)
    assert e.value.status == B.ECAPACITY


def _chunk(L, ctx, new, rows):
    """Keys, values and queries of the chunk as device buffers of `rows` rows (zeros behind the last token) and its bounds."""
    import torch
    def bits16(parts, heads):
        x = np.zeros((rows, heads, 128), np.float32)
        x[:sum(new)] = np.concatenate(parts)
        return torch.from_numpy(W.f32_to_bf16_bits(x).view(np.int16)).cuda()
    n = range(len(new))
    K = bits16([L.tokens[b][0][ctx[b]:ctx[b] + new[b]] for b in n], L.wl.n_kv)
    V = bits16([L.tokens[b][1][ctx[b]:ctx[b] + new[b]] for b in n], L.wl.n_kv)
    Q = bits16([L.wl.chunk_queries(b, np.arange(ctx[b], ctx[b] + new[b])) for b in n], L.wl.n_q)
    return K, V, Q, torch.tensor([0] + list(np.cumsum(new)), dtype=torch.int32, device="cuda")


@pytest.mark.parametrize("word", [0x00, 0x40, 0x4E, 0xFF])      # as counts of shares: 0, 3.0, 8.6e8, not a number
def test_rows_without_a_sequence_are_left_alone(word):
    """total_new above cu_new[batch] (a buffer padded to a fixed size): whatever the workspace held for the rows behind the last
    sequence, they are not written and the others are right."""
    import torch
    from paper_2609_38121_b200 import binding as B
    ctx, new, rows = [1200, 300], [20, 40], 67
    L = Layer(_wl(8, 2, 2), [c + n for c, n in zip(ctx, new)], 2, 4, 64, 1)
    L.append_step(ctx)
    L.prefill(new)
    full = L.first
    K, V, Q, cu = _chunk(L, ctx, new, rows)
    nbytes = B.prefill_workspace_bytes(L.cache.desc, 2, rows)
    ws = torch.full((nbytes,), word, dtype=torch.uint8, device="cuda")
    O = torch.full((rows, 8, 128), float("nan"), device="cuda")
    B.prefill_attn(L.cache.desc, 2, L.slot, L.seq_len, cu, rows, 40, K, V, Q, O, ws, nbytes)
    out = O.cpu().numpy()
    assert L.cache.status() == 0
    assert np.all(np.isnan(out[60:]))
    assert np.max(np.abs(out[:60] - full)) <= 1e-3 * np.max(np.abs(full))


@pytest.mark.parametrize("with_table", [True, False])
def test_more_tokens_than_promised(with_table):
    """A sequence with more new tokens than max_new: its rows past the tile pairs of max_new tokens have no output, and that is reported."""
    import torch
    from paper_2609_38121_b200 import binding as B
    ctx, new = [1200, 300], [20, 200]
    L = Layer(_wl(8, 2, 2), [c + n for c, n in zip(ctx, new)], 2, 4, 64, 1)
    L.append_step(ctx)
    L.prefill(new)
    full = L.first
    K, V, Q, cu = _chunk(L, ctx, new, 220)
    nbytes = B.prefill_workspace_bytes(L.cache.desc, 2, 220)
    if not with_table:                                  # 8 pairs over the two KV heads: 16 shares at most, behind the operands
        up = lambda x: (x + 255) // 256 * 256  # noqa: E731
        nbytes = up(2 * up(220 * 2 * 256) + up(2 * 220 * 8 * 256) + up(220 * 8 * 4) + 16 * 220 * 8 * 528)
    ws = torch.full((nbytes,), 0x40, dtype=torch.uint8, device="cuda")
    O = torch.full((220, 8, 128), float("nan"), device="cuda")
    B.prefill_attn(L.cache.desc, 2, L.slot, L.seq_len, cu, 220, 64, K, V, Q, O, ws, nbytes)
    out = O.cpu().numpy()
    assert L.cache.status() == B.DEV_BAD_COUNT
    assert np.all(np.isnan(out[20 + 64:]))              # one pair of 32-position tiles per sequence
    assert np.max(np.abs(out[:84] - full[:84])) <= 1e-3 * np.max(np.abs(full))


@pytest.mark.parametrize("ctx,new,n_q,n_kv,shares", [
    ([1200, 300], [20, 40], 8, 2, 16),                  # two pairs per KV head: as many shares as the workspace holds
    ([2368], [2368], 8, 1, 2),                          # 74 pairs of one KV head: two shares fill 148 SMs once
])
def test_least_workspace_holds_one_wave(ctx, new, n_q, n_kv, shares):
    """The least workspace that is accepted holds one wave of shares, and the call makes use of all of them: the number that it
    leaves beside the partial results of every row (behind the operands; rows of 132 floats, the count is the last but one)."""
    import torch
    from paper_2609_38121_b200 import binding as B
    if torch.cuda.get_device_properties(0).multi_processor_count != 148:
        pytest.skip("counts of a GPU with 148 SMs")
    total = sum(new)
    L = Layer(_wl(n_q, n_kv, len(ctx)), [c + n for c, n in zip(ctx, new)], 2, 4, 64, 1)
    L.append_step(ctx, oracle_too=False)
    L.append_step(new, oracle_too=False)
    K, V, Q, cu = _chunk(L, ctx, new, total)
    up = lambda x: (x + 255) // 256 * 256  # noqa: E731
    operands = 2 * up(total * n_kv * 256) + up(2 * total * n_q * 256) + up(total * n_q * 4)
    least, asked = up(operands + shares * total * n_q * 528), B.prefill_workspace_bytes(L.cache.desc, len(ctx), total)
    outs = []
    for nbytes in (least, asked):
        ws = torch.zeros(nbytes, dtype=torch.uint8, device="cuda")
        O = torch.full((total, n_q, 128), float("nan"), device="cuda")
        B.prefill_attn(L.cache.desc, len(ctx), L.slot, L.seq_len, cu, total, max(new), K, V, Q, O, ws, nbytes)
        outs.append(O.cpu().numpy())
        counts = ws[operands:operands + total * n_q * 528].view(torch.float32).view(-1, 132)[:, 130]
        if nbytes == least:
            assert torch.all(counts == shares)
    assert np.max(np.abs(outs[0] - outs[1])) <= 1e-3 * np.max(np.abs(outs[1]))
    with pytest.raises(B.WushkvError) as e:
        B.prefill_attn(L.cache.desc, len(ctx), L.slot, L.seq_len, cu, total, max(new), K, V, Q, O, ws, least - 1)
    assert e.value.status == B.ECAPACITY
