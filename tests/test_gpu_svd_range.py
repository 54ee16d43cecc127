"""The Jacobi SVD's arithmetic at the edges of its range: rotation angles in FP64,
graded columns, exact zeros, scales, and columns too long for shared memory."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _svd(A, **kw):
    from paper_1506_05083_gb300 import axi
    At = torch.tensor(np.ascontiguousarray(A.T), device="cuda")
    V, sigma, sweeps = axi.svd_jacobi(At, **kw)
    return At, V, sigma, sweeps


def _orthonormal(m, n, seed):
    rng = np.random.default_rng(seed)
    return np.linalg.qr(rng.normal(size=(m, n)) + 1j * rng.normal(size=(m, n)))[0]


def test_svd_angles_are_fp64():
    """Two columns need one rotation, and the sweep that finds nothing left to rotate:
    with the angle to FP64 rounding the columns are orthogonal to 4 * 2^-53 after the
    first (an FP32 angle leaves 1e-8 and takes a third sweep)."""
    rng = np.random.default_rng(3)
    for _ in range(20):
        A = rng.normal(size=(6, 2)) + 1j * rng.normal(size=(6, 2))
        assert _svd(A)[3] <= 2
