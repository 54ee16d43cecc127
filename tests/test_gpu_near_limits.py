"""The near-image expansions at the limits of their rules: shared-memory grants of
calls of several sizes in one process."""
import numpy as np
import pytest

import synth

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
