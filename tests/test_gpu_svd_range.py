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


@pytest.mark.parametrize("m,n,low", [(3, 2, -20), (40, 25, -60), (90, 60, -130)])
def test_svd_graded_columns(m, n, low):
    """Orthonormal columns times powers of ten from 1 down to 10^low, in mixed order: the
    singular values are those powers and come back relative to themselves, n reflectors
    and n rotations a sweep of a few rounding units each (sqrt(11 n) 4 * 2^-53, times four)."""
    s = 10.0 ** np.linspace(0, low, n)[np.random.default_rng(n).permutation(n)]
    At, V, sigma, _ = _svd(_orthonormal(m, n, 1) * s)
    got = np.sort(sigma.cpu().numpy())
    assert np.abs(got / np.sort(s) - 1).max() < 1e-13
    Vn = V.cpu().numpy().T
    assert np.abs(Vn.conj().T @ Vn - np.eye(n)).max() < 1e-13


@pytest.mark.parametrize("scale", [1e-75, 1e-30, 1e60])
def test_svd_scaled(scale):
    """A matrix of any scale whose squares stay in range: the values of the unscaled one."""
    rng = np.random.default_rng(8)
    A = rng.normal(size=(50, 31)) + 1j * rng.normal(size=(50, 31))
    got = np.sort(_svd(A * scale)[2].cpu().numpy())[::-1] / scale
    s = np.linalg.svd(A, compute_uv=False)
    assert np.abs(got - s).max() < 1e-13 * s[0]


@pytest.mark.parametrize("zeros", [(2,), (0, 5, 6), tuple(range(1, 20))])
def test_svd_zero_columns_are_exact(zeros):
    """Zero columns give exact zeros, V stays unitary, and a solve without cutoff drops
    them: the minimum-norm least-squares solution."""
    from paper_1506_05083_gb300 import axi
    m, n = 37, 20
    rng = np.random.default_rng(2)
    A = rng.normal(size=(m, n)) + 1j * rng.normal(size=(m, n))
    A[:, list(zeros)] = 0.0
    At, V, sigma, _ = _svd(A)
    assert int((sigma == 0).sum()) == len(zeros)
    Vn = V.cpu().numpy().T
    assert np.abs(Vn.conj().T @ Vn - np.eye(n)).max() < 1e-13
    b = rng.normal(size=(2, m)) + 1j * rng.normal(size=(2, m))
    x = axi.svd_solve(At, V, sigma, torch.tensor(b, device="cuda"), 0.0).cpu().numpy()
    keep = [j for j in range(n) if j not in zeros]
    want = np.zeros((n, 2), dtype=complex)
    want[keep] = np.linalg.lstsq(A[:, keep], b.T, rcond=None)[0]
    cond = np.linalg.cond(A[:, keep])
    assert np.abs(x.T - want).max() < 1e-13 * cond ** 2 * np.abs(want).max()


@pytest.mark.parametrize("m,n,kind", [(7100, 12, "full"), (7060, 9, "zero"), (7090, 10, "graded")])
def test_svd_long_columns(m, n, kind):
    """n + m above the shared memory of a block pair: rounds of single pairs in global
    memory and the permutation by cycles."""
    rng = np.random.default_rng(m)
    A = rng.normal(size=(m, n)) + 1j * rng.normal(size=(m, n))
    s = None
    if kind == "zero":
        A[:, [0, 4]] = 0.0
    if kind == "graded":
        s = 10.0 ** np.linspace(-90, 0, n)
        A = _orthonormal(m, n, 4) * s
    At, V, sigma, _ = _svd(A)
    US, Vn, sg = At.cpu().numpy().T, V.cpu().numpy().T, sigma.cpu().numpy()
    ref = np.sort(np.linalg.svd(A, compute_uv=False) if s is None else s)
    assert np.abs(np.sort(sg) - ref).max() < 1e-13 * ref[-1]
    if kind == "zero":
        assert int((sg == 0).sum()) == 2
    if kind == "graded":
        assert np.abs(np.sort(sg) / ref - 1).max() < 1e-13
    assert np.abs(Vn.conj().T @ Vn - np.eye(n)).max() < 1e-13
    assert np.abs(US @ Vn.conj().T - A).max() < 1e-13 * ref[-1]


@pytest.mark.parametrize("N,P", [(1, 4), (2, 8), (13, 8), (23, 40), (24, 40)])
def test_tsvd_small_blocks(N, P):
    """Truncated-SVD blocks on either side of the width from which they are a batch:
    test_tsvd_blocks's checks and tolerances."""
    import test_gpu_svd_blocks as blocks
    blocks.test_tsvd_blocks(N, P)
