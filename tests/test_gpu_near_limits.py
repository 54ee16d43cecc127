"""The near-image expansions at the limits of their rules: shared-memory grants of
calls of several sizes in one process, lattices whose images are far away, and
large k r."""
import numpy as np
import pytest

import synth
from test_gpu_near_sph import _abs_sum

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _operator(N, P, k, M=None):
    from paper_1506_05083_gb300 import axi
    ob = synth.small_case(seed=31, k=k, M=M or int(np.ceil(1.2 * N)), N=N, P=P).obstacles[0]
    return axi.Operator([axi.spec_from_obstacle(ob)])


def test_near_sizes_one_after_another():
    """Degrees p near 113 (tables of 51 KB, eight waves a tile) and 80 (37 KB, tiles of
    one, two and four): the first small call of a tile must not lower the limit that
    the large one had set. A call returns the same bits before and after the others."""
    from paper_1506_05083_gb300 import axi
    N, P = 40, 34
    op = _operator(N, P, 6.0)
    rng = np.random.default_rng(0)
    c = torch.tensor(rng.standard_normal((9, P, N)) + 1j * rng.standard_normal((9, P, N)), device="cuda")
    d = torch.tensor(synth.plane_wave_directions(9, 3), device="cuda")
    near = lambda W, lat: axi.near_image_sum(op, c[:W].contiguous(), (lat, lat), d[:W].contiguous(), slices=7)  # noqa: E731
    large = near(9, 2.78)
    for W in (1, 2, 4):
        small = near(W, 3.1)
        assert torch.equal(near(9, 2.78), large), W
        assert torch.equal(near(W, 3.1), small), W


def _against_direct(op, k, lat, c, slices):
    """Error of a split call against the direct FP64 sum, relative to sum |K| |sigma|."""
    from paper_1506_05083_gb300 import axi
    spec = op.specs[0]
    d = torch.tensor(synth.plane_wave_directions(c.shape[0], 3), device="cuda")
    ct = torch.tensor(c, device="cuda")
    ref = axi.near_image_sum(op, ct, lat, d, slices=0)
    U = axi.near_image_sum(op, ct, lat, d, slices=slices)
    return (U - ref).abs().max().item() / _abs_sum(k, spec.coll, spec.src, c[:, :, :spec.N], lat, spec.P)


@pytest.mark.parametrize("lat", [(30.0, 30.0), (3.0e3, 3.0e3), (2.0e5, 9.0e4), (4.0, 1.0e5), (2.0e6, 2.0e6)])
def test_near_far_lattices(lat):
    """Periods from ten to a million body sizes, where h_l(k D) runs upwards (k D beyond
    every degree) and beyond k D = 2^19, where the direct split sum serves. Tolerance: that
    of the other lattices, 1.5e-13, and the phases: k, D and R enter both sums with four
    roundings of k D radians."""
    k, N, P = 3.0, 30, 18
    op = _operator(N, P, k)
    rng = np.random.default_rng(5)
    c = rng.standard_normal((2, P, N)) + 1j * rng.standard_normal((2, P, N))
    err = _against_direct(op, k, lat, c, 7)
    assert err < 1.5e-13 + 4 * 2.0 ** -53 * k * np.hypot(*lat), err


@pytest.mark.parametrize("kr,slices", [(34.0, 7), (44.5, 7), (57.0, 7), (54.0, 6), (60.0, 6), (34.0, 4)])
def test_near_large_kr(kr, slices):
    """One source a wave, so that the error is relative to single kernel values: a
    split call keeps the digits it was asked for, 2^(-7 slices + 5), whether the
    expansions (whose translation loses digits as k r grows) or the direct sum serves.
    Three waves a call, where the expansions are expected to be the faster."""
    from paper_1506_05083_gb300 import axi
    N, P = 30, 18
    spec = _operator(N, P, 1.0).specs[0]
    z = np.linspace(-0.3, 0.3, 6001)                        # centre of the smallest sphere
    rad = lambda a: np.hypot(a[:, 0], a[:, 1] - z[:, None]).max(1)  # noqa: E731
    zc = np.argmin(np.maximum(rad(spec.coll), rad(spec.src)))
    rs, rt = rad(spec.src)[zc], rad(spec.coll)[zc]
    k, D = kr / rt, 1.3 * (rs + rt)
    op = axi.Operator([axi.ObstacleSpec(spec.bc, spec.M, N, P, spec.q, k, 0.0, spec.coll, spec.src)])
    worst = 0.0
    for j in range(0, N, 3):
        c = np.zeros((3, P, N), dtype=complex)
        for w in range(3):
            c[w, :, j + w] = 1.0                            # all modes alike: the ring's node at angle 0
        worst = max(worst, _against_direct(op, k, (D, D), c, slices))
    print(f"k r {kr}, {slices} digits: {worst:.2e}")
    assert worst < 2.0 ** (-7 * slices + 5)


@pytest.mark.parametrize("rho", [2e-6, 1e-5, 1e-3, 0.05])
def test_near_ring_close_to_the_axis(rho):
    """Rings next to the axis with oblique normals (the tip of a cone), where the normal
    derivative has a theta part of its own size: the tolerance of the other lattices,
    1.5e-13 of sum |K| |sigma|."""
    from paper_1506_05083_gb300 import axi
    N, P, k = 30, 18, 4.0
    spec = _operator(N, P, k).specs[0]
    coll = spec.coll.copy()
    coll[0, 0] = coll[-1, 0] = rho
    coll[0, 2:] = [0.8, 0.6]
    coll[-1, 2:] = [0.6, -0.8]
    op = axi.Operator([axi.ObstacleSpec(spec.bc, spec.M, N, P, spec.q, k, 0.0, coll, spec.src)])
    rng = np.random.default_rng(9)
    c = rng.standard_normal((3, P, N)) + 1j * rng.standard_normal((3, P, N))
    err = _against_direct(op, k, (3.4, 3.4), c, 7)
    assert err < 1.5e-13, err


def test_near_scratch_of_more_waves():
    """A scratch sized for 30 waves (which take the direct sum here) serves every smaller
    number of waves on the same lattice, whichever way they would go with their own."""
    from paper_1506_05083_gb300 import axi
    N, P, k, lat = 24, 18, 2.5, (2.85, 2.85)
    op = _operator(N, P, k)
    rng = np.random.default_rng(1)
    c = torch.tensor(rng.standard_normal((30, P, N)) + 1j * rng.standard_normal((30, P, N)), device="cuda")
    d = torch.tensor(synth.plane_wave_directions(30, 3), device="cuda")
    need = axi._near_bytes(op, 0, 30, lat, 7)
    scratch = torch.empty(need, dtype=torch.uint8, device="cuda")
    for W in (30, 17, 8, 3, 1):
        args = (op, c[:W].contiguous(), lat, d[:W].contiguous())
        U = axi.near_image_sum(*args, slices=7, scratch=scratch)
        ref = axi.near_image_sum(*args, slices=0)
        assert (U - ref).abs().max() < 2.0 ** -44 * N * P * ref.abs().max(), W
    with pytest.raises(axi.AxiError):
        axi.near_image_sum(*args, slices=7, scratch=scratch[:1 << 16])
