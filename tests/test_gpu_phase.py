"""sin and cos of k R straight from R's bits (trig::sincos_phase) over wavenumbers
and distances that reach its fixed-point form, its library form below 2^-10
table steps and the shifts between: the potential, its normal derivative and the
far field of two point sources against extended precision.

Tolerance: R and the products carry a few roundings, and a relative error u of R
moves the phase by u k R: 8 * 2^-53 (1 + k R) of the largest term."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [1e-9, 3e-6, 1e-3, 0.7, 25.0, 3.1e3, 2.0e6])
def test_phase_range(k):
    from paper_1506_05083_gb300 import axi
    spec = axi.ObstacleSpec(axi.BC_NEUMANN, 1, 1, 2, 4, k, 0.0, np.array([[1.0, 0.0, 1.0, 0.0]]), np.array([[0.5, 0.1]]))
    op = axi.Operator([spec])
    rng = np.random.default_rng(int(1000 * k) % 97)
    coef = rng.normal(size=(1, 2, 1)) + 1j * rng.normal(size=(1, 2, 1))
    T = rng.normal(size=(200, 3)) * (10.0 ** rng.uniform(-0.5, 2.5, size=(200, 1))) + np.array([0.0, 0.0, 3.0])
    n = rng.normal(size=(200, 3))
    sig = np.fft.ifft(coef[0, :, 0]).astype(np.clongdouble)
    Y = np.array([[0.5, 0.0, 0.1], [-0.5, 0.0, 0.1]], dtype=np.longdouble)
    D = T.astype(np.longdouble)[:, None] - Y[None]
    R = np.sqrt((D * D).sum(-1))
    kl = np.longdouble(k)
    four_pi = 4 * np.arccos(np.longdouble(-1.0))
    e = np.cos(kl * R) + 1j * np.sin(kl * R)
    far_arg = kl * (T.astype(np.longdouble) @ Y.T)
    want = {axi.EVAL_POTENTIAL: e / (four_pi * R),
            axi.EVAL_NORMAL_DERIV: (n[:, None] * D).sum(-1) * (1j * kl * R - 1) * e / (four_pi * R ** 3),
            axi.EVAL_FAR_FIELD: (np.cos(far_arg) - 1j * np.sin(far_arg)) / four_pi}
    ct, tt, nt = (torch.tensor(x, device="cuda") for x in (coef, T, n))
    for kind, K in want.items():
        got = op.eval_field(ct, tt, kind, normals=nt).cpu().numpy()[0]
        ref = (K * sig[None]).sum(-1)
        scale = (np.abs(K) * np.abs(sig)[None]).sum(-1)
        if kind == axi.EVAL_NORMAL_DERIV:                     # n . (x - y) may cancel
            scale = (np.abs(sig)[None] * np.linalg.norm(n, axis=1)[:, None] * R * np.abs(1j * kl * R - 1)
                     / (four_pi * R ** 3)).sum(-1)
        arg = np.abs(far_arg).max(-1) if kind == axi.EVAL_FAR_FIELD else (kl * R).max(-1)
        if kind == axi.EVAL_FAR_FIELD:                        # x . y may cancel too
            arg = kl * 0.51 * np.linalg.norm(T, axis=1)
        err = np.abs(got - ref) / scale
        assert np.all(err <= 8 * 2.0 ** -53 * (1 + arg)), (kind, float((err / (1 + arg)).max()))
