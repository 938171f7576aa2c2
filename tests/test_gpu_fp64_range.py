"""FP64 fronts near the ends of FP64's range: a matrix times a power of two has the same
factors, scaled, as long as its entries stay in range; Schur products may be subnormal or
lie in the last binade."""
import numpy as np
import pytest

import synth
from oracle.rsd_exact import lu_nopivot

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rsd():
    from paper_1210_6266_gb300 import build
    build.build()
    import paper_1210_6266_gb300 as m
    return m


def _setup(rsd, A, owner, **kw):
    nz = A != 0.0
    p = rsd.RSD_PREC_FP64
    return rsd.RSD.setup(torch.as_tensor(np.concatenate([[0], nz.sum(1).cumsum()]).astype(np.int64), device="cuda"),
                         torch.as_tensor(np.nonzero(nz)[1].astype(np.int32), device="cuda"),
                         torch.as_tensor(A[nz], device="cuda"), torch.as_tensor(owner, device="cuda"),
                         np.array([-1, 0], dtype=np.int32), prec_leaf=p, prec_mid=p, prec_root=p, **kw)


# diagonal entries between 2^7 and 2^8, others below 1
@pytest.mark.parametrize("power", [-1012, -500, 0, 1010])
@pytest.mark.parametrize("lu", [False, True])
def test_fp64_fronts_scaled_as_a_whole(rsd, power, lu):
    s, s_root = 200, 70
    n = s + s_root
    A = synth.uniform(8100, n * n).reshape(n, n)
    if not lu:
        A = 0.5 * (A + A.T)
    A[np.arange(n), np.arange(n)] = 1.25 * (np.abs(A).sum(1) + 1.0)
    h = _setup(rsd, np.ldexp(A, power), np.array([1] * s + [0] * s_root, dtype=np.int32), nonsymmetric=lu)
    tol = 40 * (s + s_root) * 2.2e-16
    if lu:
        L, U = lu_nopivot(A)
        d = np.abs(U).max()
        gl, gu = h.front_factor(1), np.ldexp(h.front_factor_upper(1), -power)
        assert np.abs(gl - L[:, :s]).max() <= tol and np.abs(gu - U[:s].T).max() <= tol * d
        assert np.abs(h.front_factor(0) - L[s:, s:]).max() <= tol
        assert np.abs(np.ldexp(h.front_factor_upper(0), -power) - U[s:, s:].T).max() <= tol * d
    else:
        L = np.linalg.cholesky(A)
        d = np.sqrt(np.diag(A))
        assert np.abs((np.ldexp(h.front_factor(1), -power // 2) - L[:, :s]) / d[:, None]).max() <= tol
        assert np.abs((np.ldexp(h.front_factor(0), -power // 2) - L[s:, s:]) / d[s:, None]).max() <= tol
    h.close()


def test_fp64_schur_product_in_the_last_binade(rsd):
    """130 couplings whose squares add up to 1.198 2^1023 against 1.9 2^1023: in range, and
    so is the difference."""
    s, c = 130, 1.0859375
    A = np.zeros((s + 1, s + 1))
    A[np.arange(s), np.arange(s)] = 4.0
    A[s, :s] = A[:s, s] = 2.0 * np.ldexp(c, 508)
    A[s, s] = np.ldexp(1.9, 1023)
    h = _setup(rsd, A, np.array([1] * s + [0], dtype=np.int32))
    assert np.array_equal(h.front_factor(1)[s], np.full(s, np.ldexp(c, 508)))
    # one rounding of each term and of the difference, 2^-53 of 1.9, beside the root's own
    want = np.sqrt(2.0 * (1.9 - s * c * c / 128.0)) * 2.0 ** 511
    assert abs(h.front_factor(0)[0, 0] - want) <= 8 * 2.0 ** -53 * want
    h.close()
