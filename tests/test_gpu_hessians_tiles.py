"""Attention-aware Hessians at the edges of the kernels' tiles (16 and 64 positions, 10 pairs per chunk, d_model no multiple of 16)
for the group sizes with one, two and three chunks of pairs, against the oracle's literal Jacobian form."""
import numpy as np
import pytest

from oracle import wushkv_oracle as O
from paper_2609_38121_b200 import workloads as W
from tests.test_gpu_hessians import TOL, _gpu, _inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_q,n_kv,n_tok,d_model", [(2, 1, 1, 32), (4, 2, 65, 20), (5, 1, 33, 32), (6, 1, 17, 48), (8, 1, 66, 16), (1, 1, 130, 8)])
def test_tile_edges(n_q, n_kv, n_tok, d_model):
    wl, K, Q, V, WO = _inputs(n_q, n_kv, n_tok, d_model, seed=71)
    tau = float(np.sqrt(128))
    HK, HV = _gpu(K, Q, V, WO, tau)
    G = n_q // n_kv
    for h in range(n_kv):
        rk, rv = O.attention_hessians(Q[:, h * G:(h + 1) * G], K[:, h], V[:, h], WO[h * G:(h + 1) * G], tau)
        if n_tok > 1:                                   # one position attends to itself only: v - o = 0
            assert np.max(np.abs(HK[h] - rk)) <= TOL * np.max(np.abs(rk))
        assert np.max(np.abs(HV[h] - rv)) <= TOL * np.max(np.abs(rv))


@pytest.mark.parametrize("n_q,n_kv,n_tok", [(8, 2, 510), (2, 2, 500), (3, 1, 200)])
def test_runs_agree_bit_for_bit(n_q, n_kv, n_tok):
    """Sums over several slices of positions are added in a fixed order."""
    wl, K, Q, V, WO = _inputs(n_q, n_kv, n_tok, 16, seed=73)
    first = _gpu(K, Q, V, WO, float(np.sqrt(128)))
    assert np.array_equal(first[0], first[0].transpose(0, 2, 1))
    for _ in range(5):
        again = _gpu(K, Q, V, WO, float(np.sqrt(128)))
        assert np.array_equal(first[0], again[0]) and np.array_equal(first[1], again[1])


@pytest.mark.parametrize("n_q,n_kv,n_tok", [(1, 1, 500), (3, 1, 300), (8, 1, 200)])
def test_positions_are_summed_in_float64(n_q, n_kv, n_tok):
    """Channel 5 of the queries is repeated in channel 9 at even positions and in channel 70 at odd ones (zero otherwise), so that
    every position contributes the same fp32 number to H_K[5][5] as to H_K[5][9] or H_K[5][70], and nothing to the other:
    H_K[5][5] = H_K[5][9] + H_K[5][70] up to the float64 rounding of n_tok sums.  Any fp32 sum over positions breaks this at 1e-8."""
    wl, K, Q, V, WO = _inputs(n_q, n_kv, n_tok, 16, seed=79)
    Q = Q.copy()
    Q[:, :, 9] = np.where(np.arange(n_tok)[:, None] % 2 == 0, Q[:, :, 5], 0)
    Q[:, :, 70] = np.where(np.arange(n_tok)[:, None] % 2 == 1, Q[:, :, 5], 0)
    HK, _ = _gpu(K, Q, V, WO, float(np.sqrt(128)))
    assert HK[0, 5, 9] != 0 and HK[0, 5, 70] != 0
    assert abs(HK[0, 5, 5] - HK[0, 5, 9] - HK[0, 5, 70]) <= n_tok * 2.0 ** -52 * abs(HK[0, 5, 5])


def test_seven_heads_and_a_long_sequence():
    """Three chunks of pairs, the last one short (28 pairs), and one head over many slices, against the literal form."""
    for n_q, n_tok, d_model in [(7, 70, 16), (1, 400, 8)]:
        wl, K, Q, V, WO = _inputs(n_q, 1, n_tok, d_model, seed=71)
        tau = float(np.sqrt(128))
        HK, HV = _gpu(K, Q, V, WO, tau)
        rk, rv = O.attention_hessians(Q, K[:, 0], V[:, 0], WO, tau)
        assert np.max(np.abs(HK[0] - rk)) <= TOL * np.max(np.abs(rk))
        assert np.max(np.abs(HV[0] - rv)) <= TOL * np.max(np.abs(rv))


@pytest.mark.parametrize("n_q,n_kv,n_tok,d_model", [(4, 1, 129, 33), (3, 1, 257, 7), (8, 1, 161, 15), (5, 1, 128, 16), (2, 1, 127, 31), (12, 3, 33, 17)])
def test_tensor_core_products(n_q, n_kv, n_tok, d_model):
    """Edges of the tiles of 128 keys and of 16, 32 and 128 positions, chunks of 1 to 9 pairs, odd d_model (rows of W_O that do not start
    on 8 bytes).  Three bf16 terms keep 24 bits of an operand, so what is left is fp32 summation: at most 2 (128 + 24) 2^-24 = 1.8e-5 of a
    product's largest term for the two chained contractions."""
    wl, K, Q, V, WO = _inputs(n_q, n_kv, n_tok, d_model, seed=83)
    tau = float(np.sqrt(128))
    HK, HV = _gpu(K, Q, V, WO, tau)
    G = n_q // n_kv
    for h in range(n_kv):
        rk, rv = O.attention_hessians(Q[:, h * G:(h + 1) * G], K[:, h], V[:, h], WO[h * G:(h + 1) * G], tau)
        assert np.max(np.abs(HK[h] - rk)) <= 1.8e-5 * np.max(np.abs(rk)), np.max(np.abs(HK[h] - rk)) / np.max(np.abs(rk))
        assert np.max(np.abs(HV[h] - rv)) <= 1.8e-5 * np.max(np.abs(rv)), np.max(np.abs(HV[h] - rv)) / np.max(np.abs(rv))


@pytest.mark.parametrize("tau", [1e42, 1e46, 1e300, float("inf")])
def test_temperatures_beyond_the_fp32_range(tau):
    """The probabilities are uniform, as at 1e30; 2 / tau^2 leaves next to nothing of H_K (1 / tau is a number of fp32 and becomes 0)."""
    wl, K, Q, V, WO = _inputs(4, 1, 150, 16, seed=89)
    ref, got = _gpu(K, Q, V, WO, 1e30), _gpu(K, Q, V, WO, tau)
    assert np.max(np.abs(got[1] - ref[1])) <= TOL * np.max(np.abs(ref[1]))
    assert np.max(np.abs(got[0])) <= 1e-60


def test_gamma_between_the_largest_numbers_of_bf16_and_fp32():
    """Gamma[3][3] = 3.3989e38 rounds to infinity in bf16; with small values everything else is far inside the range."""
    wl, K, Q, V, WO = _inputs(1, 1, 150, 16, seed=91)
    WO = np.zeros_like(WO)
    WO[0, 3, 5] = np.float32(1.8436e19)
    assert 3.3962e38 < float(WO[0, 3, 5]) ** 2 < 3.4028e38
    V = W.bf16_round_f32(V * np.float32(1e-4))
    tau = float(np.sqrt(128))
    HK, HV = _gpu(K, Q, V, WO, tau)
    rk, rv = O.attention_hessians(Q, K[:, 0], V[:, 0], WO, tau)
    assert np.max(np.abs(HK[0] - rk)) <= TOL * np.max(np.abs(rk))
    assert np.max(np.abs(HV[0] - rv)) <= TOL * np.max(np.abs(rv))
