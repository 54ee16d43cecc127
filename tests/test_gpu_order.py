"""The start of the trailing updates of a directly launched build, chosen by the number
of modes: a plan on either side of the rule gives the bits of the late start that
rest_start 1 asks for (the order of launches changes no result)."""
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("split", [False, True])
@pytest.mark.parametrize("P", [16, 58, 60, 62, 90])          # 9 to 46 modes; a fifth of 152 SMs is 30
def test_order_by_modes_is_exact(P, split):
    from paper_1506_05083_gb300 import axi
    ob = synth.small_case(seed=3, k=4.0, M=78, N=65, P=P).obstacles[0]
    prec = axi.PREC_SPLIT_BF16 if split else axi.PREC_FP64
    d = torch.tensor(synth.plane_wave_directions(2, 1), device="cuda")
    out = []
    for tuning in ('{"rest_start": 0}', '{"rest_start": 1}'):
        op = axi.Operator([axi.spec_from_obstacle(ob)], prec=prec, tuning=tuning)
        op.refactor()
        out.append(op.apply(op.incident(d)))
        assert op.status() == 0
    assert torch.equal(out[0], out[1])
