"""Segmented steps as chains of overlapping launches: the same bits as one
launch, also over more segments than a chain holds and from a captured
stream, and work queued behind the step finds all of its results."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_1110_4903_gb300 import chem, synth
    return torch, chem, synth


# segments of one cell, of a part of a warp, more than 64 of them (a second
# chain), a ragged last one, and one of more than four waves
@pytest.mark.parametrize("name,mixed,n,seg", [
    ("h2air-1M", False, 70, 1), ("h2air-1M", True, 3001, 37), ("h2air-1M", True, 200000, 120000),
    ("hc36-256k", True, 900, 13), ("hc36-256k", False, 400, 399)])
def test_chain_equals_one_launch(env, name, mixed, n, seg):
    torch, chem, synth = env
    mech, field, dt = synth.workload(name)
    f = synth.subsample(field, np.arange(n))
    dev = torch.device("cuda")
    ch = chem.Chem(mech, precision=chem.MIXED if mixed else chem.FP64)
    rho0 = torch.empty((mech.ns, n), dtype=torch.float64, device=dev)
    e0 = torch.empty(n, dtype=torch.float64, device=dev)
    ch.state_from_tpy(torch.tensor(f.T, device=dev), torch.tensor(f.P, device=dev),
                      torch.tensor(f.Y, device=dev), rho0, e0)
    ref, eref = rho0.clone(), e0.clone()
    st_ref = torch.full((n,), -1, dtype=torch.int32, device=dev)
    ch.advance(ref, eref, dt, status=st_ref)
    rho, e = torch.empty_like(rho0), torch.empty_like(e0)
    st = torch.empty_like(st_ref)
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    for _ in range(3):
        with torch.cuda.stream(stream):
            rho.copy_(rho0)
            e.copy_(e0)
            st.fill_(-1)
            ch.advance_segmented(rho, e, dt, seg, status=st)
            after, eafter, sta = rho.clone(), e.clone(), st.clone()   # no synchronisation in between
        stream.synchronize()
        assert torch.equal(after, ref) and torch.equal(eafter, eref) and torch.equal(sta, st_ref)
    graph = torch.cuda.CUDAGraph()
    rho.copy_(rho0)
    e.copy_(e0)
    torch.cuda.synchronize()
    with torch.cuda.graph(graph):
        ch.advance_segmented(rho, e, dt, seg, status=st)
    assert torch.equal(rho, rho0)
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(rho, ref) and torch.equal(e, eref) and torch.equal(st, st_ref)
    ch.close()
