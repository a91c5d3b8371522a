"""The transform builder on statistics at the edges of its arithmetic, against the oracle's eigensolver: very differently scaled
M and H, strongly graded spectra, repeated eigenvalues, many heads in one call, and matrices that are not positive definite."""
import numpy as np
import pytest

from oracle import wushkv_oracle as O
from paper_2609_38121_b200 import workloads as W

pytestmark = pytest.mark.gpu


def _spd(rng, spread, scale):
    q = np.linalg.qr(rng.standard_normal((128, 128)))[0]
    m = (q * (scale * 10.0 ** np.linspace(-spread, 0, 128))) @ q.T
    return 0.5 * (m + m.T)


def _build(M, H, gamma):
    import torch
    from paper_2609_38121_b200 import binding as B
    T, Ti = B.build_transforms_device(torch.from_numpy(M).cuda(), torch.from_numpy(H).cuda(), gamma)
    return T.cpu().numpy().astype(np.float64), Ti.cpu().numpy().astype(np.float64)


@pytest.mark.parametrize("m_scale,h_scale,spread", [(1.0, 1.0, 3.0), (1e20, 1e-15, 3.0), (1e-18, 1e12, 6.0)])
def test_scales_and_graded_spectra(m_scale, h_scale, spread):
    rng = np.random.default_rng(5)
    M = np.stack([_spd(rng, spread, m_scale) for _ in range(20)])
    H = np.stack([_spd(rng, spread, h_scale) for _ in range(20)])
    T, Ti = _build(M, H, W.GAMMA)
    ref, _ = O.build_transforms(M, H, W.GAMMA)
    # Both sides round the same float64 matrix to bf16: entries differ by one unit in the last place where the solvers' last bits
    # cross a rounding boundary, about (solver error / 2^-8) of them; an entry near zero differs by the solvers' error.
    unit = np.maximum(np.abs(ref), 1e-9 * np.abs(ref).max()) * 2.0 ** -7
    assert np.all(np.abs(T - ref) <= unit) and np.mean(T != ref) < 1e-3
    for h in range(20):
        np.testing.assert_allclose(Ti[h].T @ T[h], np.eye(128), atol=1e-4)


def test_repeated_eigenvalues():
    """M = H = I: any orthonormal basis diagonalises A, so T is compared through what defines it: T^T T = c^2 / 128^0 * I up to bf16."""
    T, Ti = _build(np.eye(128)[None], np.eye(128)[None].copy(), 0.0)
    g = T[0].T @ T[0]
    np.testing.assert_allclose(g, g[0, 0] * np.eye(128), atol=2.0 ** -6 * g[0, 0])
    np.testing.assert_allclose(Ti[0].T @ T[0], np.eye(128), atol=1e-4)


@pytest.mark.parametrize("which", ["hessian", "gram"])
def test_indefinite_statistics_are_refused(which):
    from paper_2609_38121_b200 import binding as B
    rng = np.random.default_rng(6)
    good, bad = _spd(rng, 2.0, 1.0), _spd(rng, 2.0, 1.0)
    bad -= 0.5 * np.eye(128)                            # eigenvalues on both sides of zero
    M, H = (good, bad) if which == "hessian" else (bad, good)
    with pytest.raises(B.WushkvError) as e:
        _build(M[None].copy(), H[None].copy(), 0.0)
    assert e.value.status == B.ENOTPD


@pytest.mark.parametrize("gamma", [0.0, 1e-8])
def test_columns_of_very_different_length(gamma):
    """Spectra of M and H over seven decades each and next to no damping: the columns that the Jacobi rotates then differ in length by
    1e6, and the tangent of their angle is the reciprocal of numbers whose square is beyond the fp32 range.  A pair that counts
    as rotated without being turned would keep the sweeps going to their limit of 30; 10 to 12 are enough (a numpy model of
    the same rule)."""
    import torch
    from paper_2609_38121_b200 import binding as B
    rng = np.random.default_rng(5)
    M, H = np.stack([_spd(rng, 7.0, 1.0) for _ in range(3)]), np.stack([_spd(rng, 7.0, 1.0) for _ in range(3)])
    nbytes = B.lib.wushkv_build_transforms_workspace_bytes(3, 128)
    dev = lambda x: torch.from_numpy(x).cuda()  # noqa: E731
    Md, Hd, ws = dev(M), dev(H), torch.zeros(nbytes // 8, dtype=torch.float64, device="cuda")
    T, Ti = torch.zeros((3, 128, 128), device="cuda"), torch.zeros((3, 128, 128), device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    stream = torch.cuda.current_stream().cuda_stream
    assert B.lib.wushkv_build_transforms_device(3, 128, Md.data_ptr(), Hd.data_ptr(), gamma, T.data_ptr(), Ti.data_ptr(), status.data_ptr(),
                                                ws.data_ptr(), nbytes, stream) == B.OK
    torch.cuda.synchronize()
    assert status.item() == 0
    sweeps = ws.view(3, 8, 128 * 128)[:, 3, 0].cpu().numpy()
    assert np.all(sweeps >= 5) and np.all(sweeps <= 16), sweeps
    ref, _ = O.build_transforms(M, H, gamma)            # compared as in test_scales_and_graded_spectra
    Td = T.cpu().numpy().astype(np.float64)
    unit = np.maximum(np.abs(ref), 1e-9 * np.abs(ref).max()) * 2.0 ** -7
    assert np.all(np.abs(Td - ref) <= unit) and np.mean(Td != ref) < 1e-3


@pytest.mark.parametrize("m_scale,h_scale,power,floor", [(1e-155, 1e-156, 512, 1e-4), (1e153, 1e153, -512, 1e-9)])
def test_statistics_at_the_ends_of_the_float64_range(m_scale, h_scale, power, floor):
    """The trace of L^T M L is 1e-310 or 1e307: its reciprocal overflows or has fewer bits.  T does not change when M and H are multiplied by
    a power of 16, so it is compared with that of the same matrices inside the range, with the tolerance of the other tests.  At the lower end
    L^T M L is summed in multiples of 2^-1074: 128 terms per entry, each rounded by up to half of that, move the matrix by about
    sqrt(128) sqrt(128) 2^-1075 = 3e-322 (2-norm).  Its eigenvalues lie between 1.7e-313 and 6e-312, the closest 2e-315 apart (numpy, the same matrices
    times 1e311), so eigenvectors turn by up to 1.5e-7; entries of T near zero differ by that much of the largest, and the floor
    allows 1e-4 2^-7 = 8e-7."""
    rng = np.random.default_rng(11)
    M, H = _spd(rng, 1.0, m_scale)[None], _spd(rng, 1.0, h_scale)[None]
    T, Ti = _build(M, H, W.GAMMA)
    ref, _ = _build(M * 2.0 ** power, H * 2.0 ** power, W.GAMMA)
    unit = np.maximum(np.abs(ref), floor * np.abs(ref).max()) * 2.0 ** -7
    assert np.all(np.abs(T - ref) <= unit) and np.mean(T != ref) < 1e-3
    np.testing.assert_allclose(Ti[0].T @ T[0], np.eye(128), atol=1e-4)
