"""Temperature recovery at and beyond the ends of its bracket, and with
negative densities: what has a temperature and what has none."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    return torch


def sensible_energy(mech, T):
    """e_s(T) less e_s(298.15 K) of every species, J/kg, [ns, len(T)]."""
    R, out = 8.314462618, []
    for a, rng, M in zip(mech.nasa7, mech.t_range, mech.molar_mass):
        def h(t):
            c = np.where((np.asarray(t) > rng[1])[..., None], a[1], a[0])
            return R / M * (sum(c[..., i] * t ** (i + 1) / (i + 1) for i in range(5)) + c[..., 5] - t)
        out.append(h(T) - h(298.15))
    return np.array(out)


@pytest.mark.parametrize("name", ["h2air-1M", "hc36-256k"])
@pytest.mark.parametrize("mixed", [False, True])
def test_recovery_beyond_the_bracket(torch, name, mixed):
    import parity as P
    from paper_1110_4903_gb300 import chem, synth
    mech, field, dt = synth.workload(name)
    rng = np.random.default_rng(11)
    f = synth.subsample(field, np.arange(600))
    # a hundredth of a kelvin to either side of the ends
    f.T[200:400] = np.where(np.arange(200) % 2, 6000.0, 200.0) + np.where(np.arange(200) % 4 < 2, 0.01, -0.01)
    rho, e = P.initial_state(mech, f)
    # energies up to far beyond those of the ends
    e[:200] += rho[:, :200].sum(0) * rng.choice([-1e9, -1e8, -1e7, 1e7, 1e8, 1e9], 200)
    # negative densities up to the size of the positive ones
    neg = rng.uniform(-1.0, 1.0, (rho.shape[0], 200)) * rho[:, 400:].sum(0)
    rho[:, 400:] = np.where(rng.uniform(size=neg.shape) < 0.3, neg, rho[:, 400:])
    ch = chem.Chem(mech, precision=chem.MIXED if mixed else chem.FP64)
    _, _, og = P.gpu_run(torch, ch, rho, e, 0.0, schedule=False)
    ch.close()
    # the oracle, where the energy has one temperature at most
    _, _, oo = P.oracle_reference(mech, rho[:, :400], e[:400], 0.0, None)
    assert np.array_equal(og["status"][:400], oo["status"])
    ok = og["status"][:400] == chem.CELL_OK
    assert 100 < ok.sum() < 300
    assert np.abs(og["T"][:400][ok] / oo["T"][ok] - 1.0).max() < 1e-12
    # the residual's signs on a grid of 1 K elsewhere: no change of sign (by
    # a thousandth of its terms, the grid's own error) means no temperature,
    # a single change upwards means one
    T = np.linspace(200.0, 6000.0, 5801)
    es = sensible_energy(mech, T)
    r = rho[:, 400:].T @ es - e[400:, None]
    tol = 1e-3 * (np.abs(rho[:, 400:]).T @ np.abs(es) + np.abs(e[400:, None])).max(1)
    total = rho[:, 400:].sum(0) > 0
    none = total & ((r.min(1) > tol) | (r.max(1) < -tol))
    up = total & (r[:, 0] < -tol) & (r[:, -1] > tol) & (np.diff(r, axis=1) > 0).all(1)
    st = og["status"][400:]
    assert none.sum() > 20 and (st[none] == chem.CELL_T_FAILED).all()
    assert (st[up] == chem.CELL_OK).all()
    for c in np.nonzero(up)[0]:
        assert abs(og["T"][400 + c] - np.interp(0.0, r[c], T)) < 1e-2


@pytest.mark.parametrize("name", ["h2air-1M", "hc36-256k"])
def test_field_temperature_from_near_and_far_guesses(torch, name):
    """A guess off by nothing, a rounding, up to the whole bracket, or none:
    the same temperature (1e-12: the energy's rounding over its slope)."""
    import parity as P
    from paper_1110_4903_gb300 import chem, synth
    mech, field, dt = synth.workload(name)
    f = synth.subsample(field, np.arange(1003))
    f.T[:8] = [200.001, 200.1, 999.999, 1000.0, 1000.001, 3000.0, 5999.9, 5999.999]
    rho, e = P.initial_state(mech, f)
    ch = chem.Chem(mech)
    dev = torch.device("cuda")
    r, ev = torch.tensor(rho, device=dev), torch.tensor(e, device=dev)
    off = np.array([0.0, 1e-16, 1e-12, 1e-9, 3e-8, 0.9e-6, 1.1e-6, 1e-4, 1e-2, 0.5, -1e-6, -1e-3, -0.7])
    guess = np.clip(f.T * (1.0 + off[np.arange(1003) % off.size]), 150.0, 7000.0)
    for g in (None, guess):
        out = torch.zeros(1003, dtype=torch.float64, device=dev)
        ch.temperature(r, ev, out, **({} if g is None else {"T_guess": torch.tensor(g, device=dev)}))
        torch.cuda.synchronize()
        assert np.abs(out.cpu().numpy() / f.T - 1.0).max() < 1e-12
    ch.close()
