"""The near-image sum by spherical-wave expansions (split sums whose lattice
keeps the images clear of the body) against the direct FP64 sum (slices 0):
P with and without the quarter turn and with a prime factor above 5, modes
folded several times over P, unequal periods (three displacement classes),
wave counts at the edges of the kernels' tiles, two-field coefficients, a body
off the origin, and a lattice too tight for the expansions.

Tolerance: every factor of the expansion (waves at sources and targets, the
two rotations, the translation) comes from recurrences of at most 127 steps,
each within a few rounding units per step, so the sum is within
5 * 127 * 2 * 2^-53 < 1.5e-13 of sum |K| |sigma|, the scale the direct sum's own
rounding is relative to; the sum of the absolute values is bounded below by
the output's own norm."""
import numpy as np
import pytest

import oracle as O
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _abs_sum(k, coll, src, coef, lattice, P):
    """max over targets and waves of sum |dG/dn| |sigma| over the eight images."""
    sig = np.abs(O.point_strengths(coef, P)).reshape(coef.shape[0], -1)
    phi = 2 * np.pi * np.arange(P) / P
    ring = lambda a, b: np.stack([a[:, None] * np.cos(phi), a[:, None] * np.sin(phi),  # noqa: E731
                                  np.broadcast_to(b[:, None], (len(a), P))], -1).reshape(-1, 3)
    X, Nv, Y = ring(coll[:, 0], coll[:, 1]), ring(coll[:, 2], coll[:, 3]), ring(src[:, 0], src[:, 1])
    B = 0.0
    for a in (-1, 0, 1):
        for b in (-1, 0, 1):
            if a or b:
                D = X[:, None] - Y[None] - np.array([a * lattice[0], b * lattice[1], 0.0])
                R = np.linalg.norm(D, axis=-1)
                B = B + sig @ (np.abs(np.einsum("tc,tsc->ts", Nv, D)) * np.abs(1j * k * R - 1) / (4 * np.pi * R ** 3)).T
    return np.max(B)


@pytest.mark.parametrize("N,P,W,k,lat,bc,shift,sph", [
    (24, 18, 5, 2.5, (3.3, 3.3), 0, 0.0, True),       # P not a multiple of 4
    (24, 22, 1, 2.5, (3.6, 3.4), 0, 0.0, True),       # P with a prime factor 11, one wave
    (30, 14, 2, 2.5, (9.0, 6.0), 0, 0.0, True),       # 2p + 1 well above P
    (33, 32, 3, 4.0, (3.7, 3.7), 0, 0.0, True),       # odd ring counts, quarter turn
    (40, 34, 9, 1.0, (5.0, 4.5), 0, 0.0, True),       # two wave tiles, the second of one wave
    (28, 30, 8, 3.0, (4.0, 4.0), 1, 0.0, True),       # transmission: two fields of coefficients
    (24, 26, 4, 2.5, (3.3, 3.3), 0, 5.0, True),       # body far above the origin
    (24, 18, 2, 2.5, (2.3, 2.3), 0, 0.0, False),      # images too close: the direct split sum
])
def test_near_expansions_vs_direct(N, P, W, k, lat, bc, shift, sph):
    from paper_1506_05083_gb300 import axi
    M = int(np.ceil(1.2 * N))
    ob = synth.small_case(seed=31, k=k, M=M, N=N, P=P, bc=bc).obstacles[0]
    coll, src, srcx = axi.geometry(ob.shape, ob.params, M, N, ob.tau)
    for a in (coll, src, srcx):
        a[:, 1] += shift
    q = axi.choose_q(M, N, P, coll, src, srcx if bc else None)
    op = axi.Operator([axi.ObstacleSpec(bc, M, N, P, q, k, 1.5 * k, coll, src, srcx if bc else None)])
    rng = np.random.default_rng(N + P)
    c = rng.standard_normal((W, P, op.specs[0].cols)) + 1j * rng.standard_normal((W, P, op.specs[0].cols))
    d = synth.plane_wave_directions(W, 3)
    ct, dt = torch.tensor(c, device="cuda"), torch.tensor(d, device="cuda")
    ref = axi.near_image_sum(op, ct, lat, dt, slices=0)
    scale = _abs_sum(k, coll, src, c[:, :, :N], lat, P)
    for slices in (6, 7):
        U = axi.near_image_sum(op, ct, lat, dt, slices=slices)
        err = (U - ref).abs().max().item() / scale
        print(f"slices {slices}: {err:.2e} of sum |K||sigma|")
        # the direct split sum keeps 7 bits a digit
        assert err < (1.5e-13 if sph else 2.0 ** (-7 * slices + 5))
    torch.cuda.synchronize()
    assert op.status() == 0
