"""FP64 fronts near the ends of FP64's range: a matrix times a power of two has the same
factors, scaled, as long as its entries stay in range; Schur products may be subnormal or
lie in the last binade.  And a symmetric matrix whose unknowns differ in scale."""
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


def test_fp64_cholesky_of_scaled_arrow_fronts(rsd):
    """Rows and columns scaled over 2^-40 .. 2^40: factors, couplings, the interface's factor
    and the application of two leaves, one of two panels, are those of the unscaled matrix, scaled."""
    sizes, s_root = [560, 140], 170
    n, r0 = sum(sizes) + s_root, sum(sizes)
    B = np.zeros((n, n))
    owner = np.zeros(n, dtype=np.int32)
    off = 0
    for c, s in enumerate(sizes):
        blk = synth.uniform(8200 + 2 * c, s * s).reshape(s, s)
        B[off:off + s, off:off + s] = 0.5 * (blk + blk.T)
        B[off:off + s, r0:] = synth.uniform(8201 + 2 * c, s * s_root).reshape(s, s_root)
        B[r0:, off:off + s] = B[off:off + s, r0:].T
        owner[off:off + s] = 1 + c
        off += s
    B[np.arange(n), np.arange(n)] = 1.25 * (np.abs(B).sum(1) + 1.0)
    e = np.round(synth.uniform(8300, n, -40.0, 40.0)).astype(int)
    A = np.ldexp(B, e[:, None] + e[None, :])
    nz = A != 0.0
    p = rsd.RSD_PREC_FP64
    h = rsd.RSD.setup(torch.as_tensor(np.concatenate([[0], nz.sum(1).cumsum()]).astype(np.int64), device="cuda"),
                      torch.as_tensor(np.nonzero(nz)[1].astype(np.int32), device="cuda"),
                      torch.as_tensor(A[nz], device="cuda"), torch.as_tensor(owner, device="cuda"),
                      np.array([-1, 0, 0], dtype=np.int32), prec_leaf=p, prec_mid=p, prec_root=p)
    S, d, rb, off = B[r0:, r0:].copy(), np.sqrt(np.diag(B)), np.arange(r0, n), 0
    for c, s in enumerate(sizes):
        rows = np.concatenate([np.arange(off, off + s), rb])
        L = np.linalg.cholesky(B[off:off + s, off:off + s])
        X = np.linalg.solve(L, B[off:off + s, r0:]).T
        got = np.ldexp(h.front_factor(1 + c), -e[rows][:, None])
        assert (np.abs(got - np.vstack([L, X])) / d[rows][:, None]).max() <= 40 * (s + 1) * 2.2e-16, c
        S -= X @ X.T
        off += s
    got = np.ldexp(h.front_factor(0), -e[rb][:, None])
    assert (np.abs(got - np.linalg.cholesky(S)) / d[rb][:, None]).max() <= 40 * (max(sizes) + s_root) * 2.2e-16
    x0 = synth.uniform(8301, n)
    z = h.apply(torch.as_tensor(np.ldexp(B @ x0, e), device="cuda"))
    assert np.abs(np.ldexp(z.cpu().numpy(), e) - x0).max() <= 1e-12
    h.close()
