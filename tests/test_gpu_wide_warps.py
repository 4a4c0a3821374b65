"""With few lanes per cell, a small call's cells and a launch's last ones are
stepped by whole warps: the same bits as a large launch gives them."""
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


def mechanism(synth, ns):
    if ns == 9:
        return synth.h2_air_9sp()
    if ns >= 13:
        return synth.hydrocarbon_mechanism(ns, 3, 3, 8 if ns < 16 else 20, 7, "m%d" % ns)
    # A + A_k <=> A_(k+1), constant cp
    nasa = np.zeros((ns, 2, 7))
    nasa[:, :, 0] = 2.5 + np.arange(ns)[:, None]
    nasa[:, :, 5] = -800.0 * np.arange(1, ns + 1)[:, None]
    nasa[:, :, 6] = 4.0 - 0.5 * np.arange(ns)[:, None]
    names = ["A%d" % (i + 1) for i in range(ns)]
    return synth.make_mechanism("chain%d" % ns, names, {a: {"H": i + 1} for i, a in enumerate(names)}, ["H"],
                                [((names[0], names[i]), (names[i + 1],), 0) for i in range(ns - 1)], nasa,
                                arr_A=[1.0e10 * (i + 1) for i in range(ns - 1)], arr_beta=[0.0, 0.5, 0.0, 0.2][:ns - 1],
                                arr_Ea=[0.0, 1.0e4, 0.0, 2.0e4][:ns - 1])


# species below, at and above multiples of the lanes per cell, up to the 31
# that leave a lane for the energy; the sizes end on both sides of the rule
# that gives each warp one cell (30 per SM), in a warp's last cells
@pytest.mark.parametrize("mixed", [False, True])
@pytest.mark.parametrize("ns,lanes", [(4, 4), (5, 4), (9, 2), (9, 4), (9, 8), (13, 8), (16, 4), (23, 8), (31, 8)])
def test_whole_warp_steps_change_nothing(env, ns, lanes, mixed):
    torch, chem, synth = env
    mech = mechanism(synth, ns)
    per_sm = 30 * torch.cuda.get_device_properties(0).multi_processor_count
    sizes = (1, 2, 32 // lanes + 1, per_sm, per_sm + 1)
    n = 3 * per_sm
    f = synth.uniform_field(ns, n, 1100.0, 2200.0, 3)
    dev = torch.device("cuda")
    ch = chem.Chem(mech, precision=chem.MIXED if mixed else chem.FP64)
    rho0 = torch.empty((ns, n), dtype=torch.float64, device=dev)
    e0 = torch.empty(n, dtype=torch.float64, device=dev)
    ch.state_from_tpy(torch.tensor(f.T, device=dev), torch.tensor(f.P, device=dev),
                      torch.tensor(f.Y, device=dev), rho0, e0)
    # (a cell without mass, one that is not a number: refused as before)
    rho0[:, 3] = 0.0
    e0[5] = float("nan")

    def step(m):
        rho, e = rho0[:, :m].clone(), e0[:m].clone()
        st = torch.full((m,), -1, dtype=torch.int32, device=dev)
        it = torch.full((m,), -1, dtype=torch.int32, device=dev)
        ch.advance(rho, e, 1e-6, status=st, newton_iters=it, lanes=lanes)
        torch.cuda.synchronize()
        return torch.cat((rho, e[None])).view(torch.int64), st, it

    ref = step(n)
    assert (ref[1] >= 0).all() and int((ref[1] == 0).sum()) > n // 2
    for m in sizes:
        for got, want in zip(step(m), ref):
            assert torch.equal(got, want[..., :m]), m
    ch.close()
