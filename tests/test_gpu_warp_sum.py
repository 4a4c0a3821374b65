"""The step kernel's sum over a warp against the exact sum of the 32 terms."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_warp_sum():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_1110_4903_gb300 import chem
    rng = np.random.default_rng(5)
    n = 20000
    same = rng.uniform(0.0, 1.0, (n, 32))
    mixed = rng.uniform(-1.0, 1.0, (n, 32))
    wide = mixed * np.exp(rng.uniform(-60.0, 0.0, (n, 32)))
    scaled = mixed * 2.0 ** rng.integers(-1000, 1000, (n, 1))
    gaps = np.where(rng.uniform(size=(n, 32)) < 0.9, 0.0, mixed)
    ends = np.array([[0.0] * 32, [-0.0] * 32, [1.0] + [0.0] * 31, [0.0] * 31 + [-1.0], [1.0, -1.0] * 16,
                     [2.0 - 2.0 ** -52] * 32, [-1.0] * 32, [2.0 ** -1000] * 32, [5e-324] * 32,
                     [1e300, -1e300] * 15 + [1e300, 1e299], [1.0] + [2.0 ** -60] * 31, [5e-324] * 31 + [3.25],
                     [1.0] * 31 + [np.inf], [1.0] * 31 + [-np.inf], [1.0] * 31 + [np.nan], [1.7e308] * 32,
                     [np.inf, -np.inf] * 16])
    x = np.concatenate([same, mixed, wide, scaled, gaps, ends])
    xd = torch.tensor(x, device="cuda")
    y = torch.empty(len(x), dtype=torch.float64, device="cuda")
    assert chem.lib().chem_selftest_warp_sum(len(x), xd.data_ptr(), y.data_ptr(), None) == 0
    y = y.cpu().numpy()
    fin = np.isfinite(x).all(1)
    fin[-2] = False   # (its sum overflows)
    # 32 terms rounded to 2^-58 of the largest, the sum to 2^-53 of itself; five
    # roundings where the tree is taken instead
    for v, s in zip(x[fin], y[fin]):
        assert abs(s - math.fsum(v)) <= 5 * 2.0 ** -53 * math.fsum(np.abs(v)) + 5e-324
    assert np.array_equal(y[-5:], np.array([np.inf, -np.inf, np.nan, np.inf, np.nan]), equal_nan=True)
