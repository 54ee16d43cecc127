"""The fill by stride classes (ring pairs on q, q/2 and q/4 nodes) against the
oracle's full-grid fill, at the edges of the split into classes: a q whose half
divides by 4, by 2 only and is odd, classes large enough to run on their own and
small enough to join a finer one, both proxy sets, native FFTs of all three
lengths, and a folded length on either side of the padding.

Tolerance: 1e-13 of max |A|, the fill's parity bar (the sub-grids agree with the
full grid to 3e-15, the eight-digit transform rounds at 2^-56 of a row)."""
import numpy as np
import pytest

import oracle as O
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp64", "split"])
@pytest.mark.parametrize("N,P,q,bc", [(30, 16, 480, 0), (30, 16, 500, 0), (30, 16, 450, 0), (48, 20, 640, 0),
                                      (90, 12, 400, 0), (26, 14, 432, 1), (64, 10, 512, 1)])
def test_fill_by_stride_class(N, P, q, bc, prec):
    from paper_1506_05083_gb300 import axi
    ob = synth.small_case(seed=9, k=2.5, M=int(np.ceil(1.2 * N)), N=N, P=P, q=q, bc=bc).obstacles[0]
    coll, src, srcx = O.geometry(ob)
    op = axi.Operator([axi.spec_from_obstacle(ob)], prec=axi.PREC_FP64 if prec == "fp64" else axi.PREC_SPLIT_BF16)
    got = op.fill_modes().cpu().numpy().transpose(0, 2, 1)
    assert op.status() == 0
    ref = O.system_matrix(ob, coll, src, srcx)
    strides = np.bincount(axi.fill_subgrid(ob.M, N, P, q, coll, src).ravel(), minlength=5)
    err = np.abs(got - ref).max() / np.abs(ref).max()
    print(f"strides 1/2/4: {strides[1]}/{strides[2]}/{strides[4]}  {err:.2e}")
    assert err <= 1e-13
