"""The mixed elimination at every size where it changes form: by columns below
24 and above 36 unknowns, in registers between, with a row to a lane up to 32
and up to four rows past those."""
import os

import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ns", [23, 24, 25, 28, 31, 32, 33, 34, 35, 36, 37])
def test_sizes_against_the_oracle(ns):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import parity as P
    from paper_1110_4903_gb300 import chem, synth
    mech = synth.hydrocarbon_mechanism(ns, 3, 3, 20, 7, "m%d" % ns)
    f = synth.uniform_field(ns, 96, 1100.0, 2200.0, 3)
    rho, e = P.initial_state(mech, f)
    ch = chem.Chem(mech, precision=chem.MIXED, lanes_per_cell=32)
    rg, eg, og = P.gpu_run(torch, ch, rho, e, 1e-6)
    ch.close()
    _, _, oo = P.oracle_reference(mech, rho, e, 1e-6, None, threads=min(16, os.cpu_count() or 1), **P.MIXED_OPTS)
    assert (og["status"] == oo["status"]).all() and (oo["status"] == 0).all()
    # every cell against the oracle along the cell's own substeps
    P.replay_check(mech, rho, e, 1e-6, None, rg, eg, og, P.TOL_MIXED, floor=P.FLOOR_MIXED)
