"""The calibration kernels at the edges of their tiles: one head and more heads than there are clusters at a time."""
import numpy as np
import pytest

from oracle import wushkv_oracle as O
from paper_2609_38121_b200 import workloads as W
from tests.test_gpu_builder import _build, _spd

pytestmark = pytest.mark.gpu


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
