"""The calibration kernels at the edges of their tiles: groups of 128 tokens and matrices that end within a thread block's part of the
list, parts of the list that go round the rings of tiles and accumulators, one head and more heads than there are clusters at a time."""
import numpy as np
import pytest

from oracle import wushkv_oracle as O
from paper_2609_38121_b200 import workloads as W
from tests.test_gpu_builder import _build, _spd

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_tok,n_q,n_kv", [(1, 1, 1), (127, 2, 1), (129, 6, 2), (128, 8, 8), (5000, 12, 4), (2561, 21, 3)])
def test_gram_sums_to_the_last_token(n_tok, n_q, n_kv):
    """Products of bf16 numbers are exact, 128 of them are summed in fp32 and the rest in float64: 2e-6 of the largest entry is the bound of
    the other Gram test.  What was in M and H before stays in the sum."""
    import torch
    from paper_2609_38121_b200 import binding as B
    gen = torch.Generator(device="cuda").manual_seed(5)
    K, Q = (torch.randn((n_tok, n, 128), generator=gen, device="cuda").to(torch.bfloat16) for n in (n_kv, n_q))
    M, H = (torch.randn((n_kv, 128, 128), generator=gen, device="cuda", dtype=torch.float64) for _ in range(2))
    k, q, G = K.double(), Q.double(), n_q // n_kv
    M_ref = M + torch.stack([k[:, h].T @ k[:, h] for h in range(n_kv)])
    H_ref = H + torch.stack([2 * sum(q[:, j].T @ q[:, j] for j in range(h * G, (h + 1) * G)) for h in range(n_kv)])
    B.accumulate_gram_device(K.view(torch.int16), Q.view(torch.int16), M, H)
    for got, ref in ((M, M_ref), (H, H_ref)):
        assert (got - ref).abs().max().item() <= 2e-6 * ref.abs().max().item()


@pytest.mark.parametrize("heads", [1, 7, 41])
def test_builder_for_one_and_for_many_heads(heads):
    rng = np.random.default_rng(heads)
    M, H = (np.stack([_spd(rng, 2.0 + h % 3, 1.0) for h in range(heads)]) for _ in range(2))
    T, Ti = _build(M, H, W.GAMMA)
    ref, _ = O.build_transforms(M, H, W.GAMMA)
    # one unit of bf16 where the solvers' last bits cross a rounding boundary, as in test_gpu_builder.py
    unit = np.maximum(np.abs(ref), 1e-9 * np.abs(ref).max()) * 2.0 ** -7
    assert np.all(np.abs(T - ref) <= unit) and np.mean(T != ref) < 1e-3
    for h in range(heads):
        np.testing.assert_allclose(Ti[h].T @ T[h], np.eye(128), atol=1e-4)


@pytest.mark.parametrize("n_tok,n_q,n_kv", [(1, 1, 1), (127, 2, 1), (32768 + 77, 7, 1)])
def test_gram_without_tensor_maps_sums_the_same(n_tok, n_q, n_kv, test_option):
    """Tiles staged by 16-byte copies: the same products.  The float64 sums are grouped alike; the CTAs' parts of a matrix meet in any order."""
    import torch
    from paper_2609_38121_b200 import binding as B
    gen = torch.Generator(device="cuda").manual_seed(6)
    K, Q = (torch.randn((n_tok, n, 128), generator=gen, device="cuda").to(torch.bfloat16).view(torch.int16) for n in (n_kv, n_q))
    sums = []
    for copies in (0, 1):
        test_option("gram_no_tma", copies)
        M, H = (torch.zeros((n_kv, 128, 128), dtype=torch.float64, device="cuda") for _ in range(2))
        B.accumulate_gram_device(K, Q, M, H)
        sums.append((M, H))
    for a, b in zip(*sums):
        assert (a - b).abs().max().item() <= 148 * 2.0 ** -52 * a.abs().max().item()


@pytest.mark.parametrize("n_tok,n_q,n_kv", [(32768 + 77, 32, 8), (65537, 7, 1), (9000, 24, 24)])
def test_gram_goes_round_its_rings(n_tok, n_q, n_kv):
    """69, 27 and 23 tiles per thread block on 148 SMs, with six places for tiles and four accumulators: every place is filled again and
    again, matrices change within a block's part, the last tile is ragged.  Bound as above."""
    import torch
    from paper_2609_38121_b200 import binding as B
    gen = torch.Generator(device="cuda").manual_seed(8)
    K, Q = (torch.randn((n_tok, n, 128), generator=gen, device="cuda").to(torch.bfloat16) for n in (n_kv, n_q))
    M, H = (torch.zeros((n_kv, 128, 128), dtype=torch.float64, device="cuda") for _ in range(2))
    B.accumulate_gram_device(K.view(torch.int16), Q.view(torch.int16), M, H)
    G = n_q // n_kv
    for h in range(n_kv):
        k = K[:, h].double()
        ref = k.T @ k
        assert (M[h] - ref).abs().max().item() <= 2e-6 * ref.abs().max().item()
        ref = sum(2 * Q[:, j].double().T @ Q[:, j].double() for j in range(h * G, (h + 1) * G))
        assert (H[h] - ref).abs().max().item() <= 2e-6 * ref.abs().max().item()


def test_builder_beyond_one_wave_of_clusters():
    """About 90 clusters of eight thread blocks run at a time; 200 heads made of five: equal statistics give equal transforms, whichever
    cluster takes them, and they are those of five heads alone."""
    rng = np.random.default_rng(13)
    M, H = (np.stack([_spd(rng, 2.0, 1.0) for _ in range(5)]) for _ in range(2))
    T, Ti = _build(M, H, W.GAMMA)
    T200, Ti200 = _build(np.tile(M, (40, 1, 1)), np.tile(H, (40, 1, 1)), W.GAMMA)
    assert np.array_equal(T200, np.tile(T, (40, 1, 1))) and np.array_equal(Ti200, np.tile(Ti, (40, 1, 1)))
