"""Segments of a state whose rows lie closer together than its cells are many
share elements: they are stepped one after another, as separate calls are."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_overlapping_rows_step_in_order():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import parity as P
    from paper_1110_4903_gb300 import chem, synth
    mech, field, dt = synth.workload("h2air-1M")
    k, segs = 256, 4
    f = synth.subsample(field, np.arange(k * segs))
    rho, e0 = P.initial_state(mech, f)
    dev = torch.device("cuda")
    # rows k apart for k * segs cells: the last cells' rows end past ns rows
    flat = torch.zeros((mech.ns + segs) * k, dtype=torch.float64, device=dev)
    flat[:mech.ns * k] = torch.tensor(np.ascontiguousarray(rho[:, :k]), device=dev).flatten()
    flat[mech.ns * k:] = torch.tensor(rho[0, :segs * k], device=dev)
    ch = chem.Chem(mech)
    ref, eref = flat.clone(), torch.tensor(e0, device=dev)
    st_ref = torch.full((k * segs,), -1, dtype=torch.int32, device=dev)
    for i in range(segs):
        c = slice(i * k, (i + 1) * k)
        ch.advance(ref[i * k:i * k + mech.ns * k].view(mech.ns, k), eref[c], dt, status=st_ref[c])
    for _ in range(3):
        got, e = flat.clone(), torch.tensor(e0, device=dev)
        st = torch.full_like(st_ref, -1)
        ch.advance_segmented(got[:mech.ns * k].view(mech.ns, k), e, dt, k, status=st)
        assert torch.equal(got.view(torch.int64), ref.view(torch.int64))
        assert torch.equal(e.view(torch.int64), eref.view(torch.int64)) and torch.equal(st, st_ref)
    ch.close()
