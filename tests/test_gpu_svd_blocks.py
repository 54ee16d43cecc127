"""The preconditioned block Jacobi SVD at the sizes where its blocks, groups of
warps and orderings change: single columns, odd counts, square and tall, one
and several column blocks, exact rank deficiency (zero columns, repeated
columns, the zero matrix), and graded columns over 1e-16.

Tolerances: U, V and U Sigma V^H come out of at most n reflectors and about ten
sweeps of n rotations a column, each unitary to a few rounding units, whose
errors add up at random: sqrt(11 n) * 4 * 2^-53 < 2.5e-14 for n <= 260; four times
that."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 1e-13


def _matrix(m, n, kind, rng):
    A = rng.normal(size=(m, n)) + 1j * rng.normal(size=(m, n))
    if kind == "graded":
        A = A @ (np.diag(10.0 ** np.linspace(0, -16, n)) @ (rng.normal(size=(n, n)) + 0j))
    elif kind == "zero_columns":
        A[:, ::3] = 0.0
    elif kind == "repeated":
        A[:, n // 2:] = A[:, :n - n // 2]
    elif kind == "zero":
        A[:] = 0.0
    return A


@pytest.mark.parametrize("m,n,kind", [(1, 1, "full"), (2, 2, "full"), (7, 3, "full"), (33, 32, "full"), (64, 64, "graded"),
                                      (200, 131, "graded"), (150, 97, "zero_columns"), (90, 60, "repeated"),
                                      (40, 17, "zero"), (700, 260, "full")])
def test_svd_shapes(m, n, kind):
    from paper_1506_05083_gb300 import axi
    A = _matrix(m, n, kind, np.random.default_rng(m + n))
    At = torch.tensor(np.ascontiguousarray(A.T), device="cuda")
    V, sigma, sweeps = axi.svd_jacobi(At)
    US, Vn, sg = At.cpu().numpy().T, V.cpu().numpy().T, sigma.cpu().numpy()
    s = np.linalg.svd(A, compute_uv=False)
    top = max(s[0], 1e-300)
    print(f"{m}x{n} {kind}: {sweeps} sweeps, sigma {np.abs(np.sort(sg)[::-1] - s).max() / top:.1e}")
    assert np.abs(np.sort(sg)[::-1] - s).max() <= TOL * top
    assert np.abs(Vn.conj().T @ Vn - np.eye(n)).max() < TOL
    assert np.abs(US @ Vn.conj().T - A).max() <= TOL * top
    keep = sg > 1e-12 * top
    U = US[:, keep] / sg[keep]
    assert np.abs(U.conj().T @ U - np.eye(keep.sum())).max() < TOL if keep.any() else np.all(US == 0.0)


def test_svd_not_finite_is_refused():
    from paper_1506_05083_gb300 import axi
    A = torch.ones(5, 9, dtype=torch.complex128, device="cuda")
    A[2, 3] = float("nan")
    with pytest.raises(axi.AxiError):
        axi.svd_jacobi(A, max_sweeps=3)


@pytest.mark.parametrize("N,P", [(24, 10), (37, 14), (61, 8)])
def test_tsvd_blocks(N, P):
    """Every mode's R = U Sigma V^H of small plans (one block pair, odd widths)."""
    import synth
    from paper_1506_05083_gb300 import axi
    ob = synth.small_case(seed=5, k=2.0, M=N + 8, N=N, P=P).obstacles[0]
    op = axi.Operator([axi.spec_from_obstacle(ob)], prec=axi.PREC_FP64 | axi.PLAN_TSVD)
    U, V, sg, sweeps = (t.cpu().numpy() for t in op.svd())
    A = op.factors()[0].cpu().numpy()
    assert op.status() == 0 and sweeps.max() < 40 and sweeps.min() >= 1
    for d in range(A.shape[0]):
        R = np.triu(A[d].T[:N])
        Ud, Vd, top = U[d].T, V[d].T, np.linalg.norm(R, 2)
        assert np.abs((Ud * sg[d]) @ Vd.conj().T - R).max() < TOL * top
        assert np.abs(Ud.conj().T @ Ud - np.eye(N)).max() < TOL
        assert np.abs(Vd.conj().T @ Vd - np.eye(N)).max() < TOL
        assert np.abs(np.sort(sg[d])[::-1] - np.linalg.svd(R, compute_uv=False)).max() < TOL * top
