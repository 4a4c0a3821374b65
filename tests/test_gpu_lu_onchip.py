"""Batched solves at the sizes where the elimination changes its threads per
system, its systems per block or its kernel: pivots, factors and (in the
interleaved layout) x bit for bit the oracle's, the contracted variant to
rounding; divisions outside the range of the corrected quotients."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_1110_4903_gb300 import chem
    return torch, chem


def _solve(env, method, A, b):
    torch, chem = env
    n_sys, n = b.shape
    dev = torch.device("cuda")
    il = method != "onchip"
    Ad = torch.tensor(np.ascontiguousarray(A.transpose(1, 2, 0)) if il else A, device=dev)
    bd = torch.tensor(np.ascontiguousarray(b.T) if il else b, device=dev)
    piv = torch.full((n_sys, n), -1, dtype=torch.int32, device=dev)
    info = torch.full((n_sys,), -1, dtype=torch.int32, device=dev)
    m = {"global": chem.LU_GLOBAL, "global_fma": chem.LU_GLOBAL_FMA, "onchip": chem.LU_ONCHIP}[method]
    chem.batched_solve(m, Ad, bd, piv, info)
    torch.cuda.synchronize()
    LU, x = Ad.cpu().numpy(), bd.cpu().numpy()
    if il:
        LU, x = LU.transpose(2, 0, 1), x.T
    return LU, x, piv.cpu().numpy(), info.cpu().numpy()


def _check(method, A, b, LU, x, piv, info, every):
    n = A.shape[1]
    eps = np.finfo(np.float64).eps
    for k in sorted(set(list(range(0, len(A), every)) + [len(A) - 1])):
        rc, LUo, pivo = oracle.lu_factor(A[k])
        assert rc == 0 and info[k] == 0
        xo = oracle.lu_solve(LUo, pivo, b[k])
        assert np.array_equal(piv[k], pivo)
        if method == "global_fma":
            assert np.abs(LU[k] - LUo).max() <= 8 * n * eps * np.abs(LUo).max()
        else:
            assert np.array_equal(LU[k], LUo)
        if method == "global":
            assert np.array_equal(x[k], xo)
        else:
            assert np.abs(x[k] - xo).max() <= 1e-13 * n * np.abs(xo).max()


# one system, a partly filled block, one system per SM and one more, more than
# the SMs hold; n around each change of the threads per system
@pytest.mark.parametrize("n,n_sys", [
    (2, 1), (8, 37), (9, 37), (9, 4864), (12, 4863), (13, 5000), (13, 78000), (14, 78000), (16, 3), (25, 153),
    (25, 6000), (26, 33), (30, 4500), (37, 1), (37, 152), (37, 2800), (41, 2500), (48, 153), (50, 1600),
    (51, 9), (56, 1217), (57, 5), (64, 152), (64, 1000), (100, 3), (100, 306), (168, 2), (169, 154), (170, 3)])
@pytest.mark.parametrize("method", ["global", "global_fma", "onchip"])
def test_sizes(env, n, n_sys, method):
    if method == "onchip" and n > 169:
        pytest.skip("does not fit on chip")
    rng = np.random.default_rng(1000 * n + n_sys)
    A = rng.standard_normal((n_sys, n, n)) + 0.5 * np.sqrt(n) * np.eye(n)[None]
    b = rng.standard_normal((n_sys, n))
    _check(method, A, b, *_solve(env, method, A, b), every=max(1, n_sys // 8))


@pytest.mark.parametrize("method", ["global", "onchip"])
@pytest.mark.parametrize("n", [14, 33, 60])
def test_divisions_outside_the_corrected_range(env, method, n):
    """Rows scaled by 2^+-450 (quotients beyond 2^+-400), entries that are
    zero, and pivots whose mantissa is all ones."""
    rng = np.random.default_rng(n)
    n_sys = 40
    A = rng.standard_normal((n_sys, n, n)) + 0.5 * np.sqrt(n) * np.eye(n)[None]
    A[:10] *= 2.0 ** rng.integers(-450, 451, (10, n, 1))
    A[10:20][rng.random((10, n, n)) < 0.3] = 0.0
    A[10:20] += np.eye(n) * 8
    A[20:30, :, 0] = rng.uniform(-0.5, 0.5, (10, n))
    A[20:30, 2, 0] = np.nextafter(1.0, 0.0)          # mantissa all ones
    A[30:] *= 2.0 ** -420
    b = rng.standard_normal((n_sys, n))
    LU, x, piv, info = _solve(env, method, A, b)
    for k in range(n_sys):
        rc, LUo, pivo = oracle.lu_factor(A[k])
        assert (rc == 0) == (info[k] == 0)
        if rc == 0:
            assert np.array_equal(piv[k], pivo) and np.array_equal(LU[k], LUo)
            if method == "global":
                assert np.array_equal(x[k], oracle.lu_solve(LUo, pivo, b[k]), equal_nan=True)


@pytest.mark.parametrize("n", [4, 14, 60])
def test_nan_and_singular_pivots_on_chip(env, n):
    rng = np.random.default_rng(n)
    A = rng.standard_normal((9, n, n)) + 0.5 * np.sqrt(n) * np.eye(n)[None]
    A[0, 0, 0] = np.nan
    A[1, 2, 0] = np.nan
    A[2, :, 1] = 0.0
    b = rng.standard_normal((9, n))
    for method in ("onchip", "global", "global_fma"):
        _, _, piv, info = _solve(env, method, A, b)
        assert piv[0, 0] == 0 and info[0] == 1
        pivo = oracle.lu_factor(A[1])[2]
        assert pivo[0] != 2 and piv[1, 0] == pivo[0] and info[1] != 0
        assert piv[2, 0] == oracle.lu_factor(A[2])[2][0] and info[2] == 2
        assert (info[3:] == 0).all()
