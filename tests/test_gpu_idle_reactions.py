"""A reaction that changes nothing does nothing, at any rate."""
import numpy as np
import pytest

import small_mechs

pytestmark = pytest.mark.gpu


# 2 A + B <=> A + 2 B (each species on both sides) behind A <=> A with a rate
# constant in FP32's range and beyond it
@pytest.mark.parametrize("mixed", [False, True])
@pytest.mark.parametrize("idle", [1e10, 1e60])
def test_rate_of_a_reaction_without_effect(idle, mixed):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import parity as P
    from paper_1110_4903_gb300 import chem, synth
    a, b = small_mechs.const_cp(3.5, -1000.0, 5.0), small_mechs.const_cp(3.5, -1000.0, 5.7)
    mech = synth.make_mechanism("idle", ["A", "B"], {"A": {"H": 1, "O": 1}, "B": {"H": 1, "O": 1}}, ["H", "O"],
                                [(("A",), ("A",), 0), (("A", "A", "B"), ("A", "B", "B"), 0)], np.stack([a, b]),
                                arr_A=[idle, 1e15], arr_beta=[0.0, 0.0], arr_Ea=[0.0, 0.0])
    f = synth.uniform_field(2, 64, 1100.0, 2200.0, 3)
    rho, e = P.initial_state(mech, f)
    ch = chem.Chem(mech, precision=chem.MIXED if mixed else chem.FP64)
    rg, eg, og = P.gpu_run(torch, ch, rho, e, 1e-6, schedule=False)
    ch.close()
    rr, er, oo = P.oracle_reference(mech, rho, e, 1e-6, None, **(P.MIXED_OPTS if mixed else {}))
    P.compare(rg, eg, og, rr, er, oo, rho, P.TOL_MIXED if mixed else P.TOL_FP64,
              floor=P.FLOOR_MIXED if mixed else P.FLOOR)
