"""Launches that do not fill the GPU: the step's blocks shrink with the cell
count, and a cell's result does not depend on the launch it is part of."""
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


# one cell, a part of a warp, one warp on every SM and one cell more, one and
# two blocks on every SM and a cell more, just below the resident slots
@pytest.mark.parametrize("name,mixed,sizes", [
    ("h2air-1M", False, (1, 7, 9, 152 * 8, 152 * 8 + 1, 152 * 80 + 1)),
    ("hc36-256k", True, (1, 33, 152, 153, 1520, 1521, 3039)),
])
def test_small_launches_equal_a_large_one(env, name, mixed, sizes):
    torch, chem, synth = env
    mech, field, dt = synth.workload(name)
    n = max(sizes) + 500
    f = synth.subsample(field, np.arange(n))
    dev = torch.device("cuda")
    ch = chem.Chem(mech, precision=chem.MIXED if mixed else chem.FP64)
    rho0 = torch.empty((mech.ns, n), dtype=torch.float64, device=dev)
    e0 = torch.empty(n, dtype=torch.float64, device=dev)
    ch.state_from_tpy(torch.tensor(f.T, device=dev), torch.tensor(f.P, device=dev),
                      torch.tensor(f.Y, device=dev), rho0, e0)

    def step(m):
        rho, e = rho0[:, :m].clone(), e0[:m].clone()
        st = torch.full((m,), -1, dtype=torch.int32, device=dev)
        it = torch.full((m,), -1, dtype=torch.int32, device=dev)
        ch.advance(rho, e, dt, status=st, newton_iters=it)
        torch.cuda.synchronize()
        return rho, e, st, it

    ref = step(n)
    assert (ref[2] >= 0).all()
    for m in sizes:
        for got, want in zip(step(m), ref):
            assert torch.equal(got, want[..., :m]), m
    ch.close()
