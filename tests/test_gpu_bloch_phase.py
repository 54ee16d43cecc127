"""C with Bloch factors whose products are 1 up to rounding: a square lattice with
|kx| = |ky| (conjugate factors multiply to 1 with an imaginary part of either sign
near 1e-17), and phases below the last bit of a table step, of either sign. Such a
phase must stay next to zero (trig::phase_offset).

Tolerance: that of the C block's parity test, 1e-12 of the block's scale (each
entry sums at most nine images, each a few roundings, and a transform of P terms)."""
import numpy as np
import pytest

import oracle as O
import synth
from oracle import periodizing as OP

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_c_near_zero_phases():
    from paper_1506_05083_gb300 import axi
    ex, ey, z0, m1 = 2.6, 2.6, 1.6, 4
    ob = synth.small_case(seed=7, k=3.0, M=24, N=20, P=16).obstacles[0]
    _, src, _ = O.geometry(ob)
    op = axi.Operator([axi.spec_from_obstacle(ob)], prec=axi.PREC_FP64)
    phases = [(s * x, t * x) for x in (1e-3, 1e-2, 0.05, 0.3, 0.7, 1.9, 3.0) for s in (1, -1) for t in (1, -1)]
    phases += [(-1e-20, 0.0), (0.0, -1e-19), (1e-20, -1e-20), (-0.0, -0.0), (3e-17, -2e-17), (np.pi, -np.pi)]
    for x, y in phases:
        cell = axi.Cell(x / ex, y / ey, ex, ey, z0, m1, 3, 4)
        G = op.c_block(cell).cpu().numpy().T
        ref = OP.c_matrix(ob, src, x / ex, y / ey, ex, ey, z0, m1)
        err = np.abs(G - ref).max() / np.abs(ref).max()
        assert err < 1e-12, (x, y, float(err))
    assert op.status() == 0
