"""Temperature recovery of species whose energy or heat capacity changes at
T_mid: the step, the field conversion and the oracle agree on what has a
temperature and on which it is."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
R, TREF, NS = 8.314462618, 298.15, 6


@pytest.fixture(scope="module")
def torch():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    return torch


class Stepped:
    """Inert species with cp/R = a1 + a2 T.  Above t_mid their heat capacity
    c_v is (1 + jump) as large, and their energy is higher by what `step`
    kelvins of c_v make at t_mid."""

    def __init__(self, step=0.0, jump=0.0, t_mid=1000.0, a2=0.0):
        from paper_1110_4903_gb300 import synth
        self.t_mid = t_mid
        nasa = np.zeros((NS, 2, 7))
        for s in range(NS):
            a1 = 2.5 + 0.5 * s
            lo = np.array([a1, a2, 0, 0, 0, -500.0 * s, 10.0])
            hi = lo.copy()
            hi[0], hi[1] = 1.0 + (a1 - 1.0) * (1.0 + jump), a2 * (1.0 + jump)
            cv = a1 - 1.0 + a2 * t_mid
            # a6: the energy at t_mid, in kelvins of R/M
            hi[5] = lo[5] + step * cv - jump * ((a1 - 1.0) * t_mid + a2 * t_mid ** 2 / 2)
            nasa[s] = lo, hi
        names = ["X%d" % s for s in range(NS)]
        self.mech = synth.make_mechanism("stepped", names, {a: {"H": s + 1} for s, a in enumerate(names)}, ["H"],
                                         [((names[0],), (names[0],), 0)], nasa, arr_A=[0.0], arr_beta=[0.0],
                                         arr_Ea=[0.0], t_mid=t_mid)
        self.a = nasa.astype(np.longdouble)

    def energies(self, T, side=None):
        """e_s(T) - e_s(298.15 K), J/kg, [species, cells], in extended precision
        (side: the range to take)."""
        T = np.asarray(T, np.longdouble)

        def e(t, rg):
            c = self.a[:, :, :, None][:, rg] if np.isscalar(rg) else \
                np.where(rg[None, None], self.a[:, 1, :, None], self.a[:, 0, :, None])
            return c[:, 0] * t + c[:, 1] * t * t / 2 + c[:, 5] - t
        M = np.asarray(self.mech.molar_mass, np.longdouble)[:, None]
        ref = e(np.longdouble(TREF), 0)
        return np.longdouble(R) / M * (e(T, (T > self.t_mid) if side is None else side) - ref)

    def densities(self, n, seed):
        return np.ascontiguousarray(np.random.default_rng(seed).dirichlet(np.ones(NS), n).T) * 0.3


def temperatures(torch, st, rho, e, guess, precision):
    """Temperature and status of a step of no length, and the field's temperature."""
    import parity as P
    from paper_1110_4903_gb300 import chem
    with_chem = chem.Chem(st.mech, precision=precision)
    _, _, og = P.gpu_run(torch, with_chem, rho, e, 0.0, T_in=guess, schedule=False)
    dev = torch.device("cuda")
    out = torch.zeros(e.size, dtype=torch.float64, device=dev)
    with_chem.temperature(torch.tensor(rho, device=dev), torch.tensor(e, device=dev), out,
                          **({} if guess is None else {"T_guess": torch.tensor(guess, device=dev)}))
    torch.cuda.synchronize()
    with_chem.close()
    return og["T"], og["status"], out.cpu().numpy()


# from a few hundredths of a kelvin to a tenth of T; few cells (a warp each)
# and many (several to a warp).  (Mixed, the largest step is left out: Newton's
# FP32 slopes take it to and fro across the step, past the recovery's 50 passes
# in a cell of a thousand.)
@pytest.mark.parametrize("n", [240, 6000])
@pytest.mark.parametrize("step,mixed", [(step, mixed) for step in (0.01, 0.02, 0.03, 0.1, 1.0, 10.0)
                                        for mixed in (False, True)] + [(100.0, False)])
def test_energy_inside_a_step(torch, step, n, mixed):
    import parity as P
    from paper_1110_4903_gb300 import chem
    st = Stepped(step=step)
    rng = np.random.default_rng(3)
    rho = st.densities(n, 4)
    lo, hi = ((rho * st.energies(np.full(n, 1000.0), side)).sum(0) for side in (0, 1))
    e = (lo + rng.uniform(0.02, 0.98, n) * (hi - lo)).astype(np.float64)
    for guess in (None, 1000.0 + rng.choice([-400.0, -1.0, -1e-3, 0.0, 1e-3, 1.0, 400.0], n)):
        T, status, field = temperatures(torch, st, rho, e, guess, chem.MIXED if mixed else chem.FP64)
        _, _, oo = P.oracle_reference(st.mech, rho, e, 0.0, guess)
        assert (oo["status"] == 0).all() and (status == 0).all()
        # (the recovery halves its bracket down to 1e-13 T)
        for t in (T, field, oo["T"]):
            assert np.abs(t / 1000.0 - 1.0).max() < 1e-12


# a heat capacity that changes by a part in 10^5 to a half at T_mid (the
# energy continuous there), and energies that step by less than a millikelvin:
# a last Newton step that crosses T_mid is no better than those differences
@pytest.mark.parametrize("mixed", [False, True])
@pytest.mark.parametrize("step,jump", [(0.0, 0.5), (0.0, -0.3), (0.0, 0.05), (0.0, 1e-5), (1e-7, 0.0), (2e-4, 0.0)])
def test_last_steps_across_t_mid(torch, step, jump, mixed):
    from paper_1110_4903_gb300 import chem
    st = Stepped(step=step, jump=jump)
    rng = np.random.default_rng(6)
    n = 6000
    rho = st.densities(n, 7)
    # to either side of T_mid by up to 2e-6 of it, guessed from as near
    sign = rng.choice([-1.0, 1.0], n)
    T0 = 1000.0 + sign * 10.0 ** rng.uniform(-8.0, -2.7, n)
    guess = 1000.0 - sign * 10.0 ** rng.uniform(-8.0, -2.7, n)
    e = (rho * st.energies(T0)).sum(0).astype(np.float64)
    for g in (guess, None):
        T, status, field = temperatures(torch, st, rho, e, g, chem.MIXED if mixed else chem.FP64)
        assert (status == 0).all()
        # (the energy's rounding over its slope, and the recovery's own 1e-13 T)
        assert np.abs(T / T0 - 1.0).max() < 1e-12 and np.abs(field / T0 - 1.0).max() < 1e-12


# energies that step down at T_mid leave two temperatures to an energy near
# there: the answer is the upper one, which the FP64 iterations meet first on
# their way down from 1500 K, also within a rounding of FP32 above T_mid
def test_energy_steps_down(torch):
    from paper_1110_4903_gb300 import chem
    st = Stepped(step=-1.0)
    rng = np.random.default_rng(8)
    for n in (240, 6000):
        rho = st.densities(n, 9)
        T0 = 1000.0 + 10.0 ** rng.uniform(-7.0, -1.0, n)
        e = (rho * st.energies(T0)).sum(0).astype(np.float64)
        T, status, field = temperatures(torch, st, rho, e, None, chem.FP64)
        assert (status == 0).all()
        assert np.abs(T / T0 - 1.0).max() < 1e-12 and np.abs(field / T0 - 1.0).max() < 1e-12


# where an energy steps by more than a thousandth of T, up or down, no guess
# is the guess 1500 K: also within a thousandth of the step's ends, where the
# recovery's passes may not suffice
@pytest.mark.parametrize("mixed", [False, True])
@pytest.mark.parametrize("step", [-20.0, 2.0, 20.0, 100.0])
def test_no_guess_is_the_plain_start(torch, step, mixed):
    from paper_1110_4903_gb300 import chem
    st = Stepped(step=step)
    rng = np.random.default_rng(12)
    n = 60000
    rho = st.densities(n, 13)
    lo, hi = ((rho * st.energies(np.full(n, 1000.0), side)).sum(0) for side in (0, 1))
    e = (lo + rng.uniform(0.0, 1.0, n) * (hi - lo)).astype(np.float64)
    cold, warm = (temperatures(torch, st, rho, e, guess, chem.MIXED if mixed else chem.FP64)
                  for guess in (None, np.full(n, 1500.0)))
    for a, b in zip(cold, warm):
        assert np.array_equal(a, b, equal_nan=True)
