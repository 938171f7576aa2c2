"""Nonsymmetric FP64 fronts whose equations and unknowns differ in scale: A = Dr B Dc with
powers of two, whose LU without pivoting is that of B, scaled (L = Dr L_B Dr^-1, U = Dr U_B Dc,
exactly).  The factors and the application, scaled back, are held to the tolerances of
the unscaled fronts."""
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


def _arrow(sizes, s_root, seed, weak):
    """Nonsymmetric diagonally dominant arrow matrix (dense leaf blocks, one dense
    interface); `weak`: unknowns of two kinds (0 / 1), coupled 2^-20 as strongly as within one."""
    n = sum(sizes) + s_root
    r0 = n - s_root
    A = np.zeros((n, n))
    owner = np.zeros(n, dtype=np.int32)
    off = 0
    for c, s in enumerate(sizes):
        A[off:off + s, off:off + s] = synth.uniform(seed + 3 * c, s * s).reshape(s, s)
        A[off:off + s, r0:] = synth.uniform(seed + 3 * c + 1, s * s_root).reshape(s, s_root)
        A[r0:, off:off + s] = synth.uniform(seed + 3 * c + 2, s * s_root).reshape(s_root, s)
        owner[off:off + s] = 1 + c
        off += s
    A[r0:, r0:] = synth.uniform(seed + 1001, s_root * s_root).reshape(s_root, s_root)
    kind = (synth.uniform(seed + 1002, n) > 0).astype(int)
    if weak:
        A *= np.where(kind[:, None] == kind[None, :], 1.0, 2.0 ** -20)
    A[np.arange(n), np.arange(n)] = 1.25 * (np.abs(A).sum(1) + 1.0)
    return A, owner, np.array([-1] + [0] * len(sizes), dtype=np.int32), kind


def _setup(rsd, A, owner, parent):
    nz = A != 0.0
    p = rsd.RSD_PREC_FP64
    return rsd.RSD.setup(torch.as_tensor(np.concatenate([[0], nz.sum(1).cumsum()]).astype(np.int64), device="cuda"),
                         torch.as_tensor(np.nonzero(nz)[1].astype(np.int32), device="cuda"),
                         torch.as_tensor(A[nz], device="cuda"), torch.as_tensor(owner, device="cuda"), parent,
                         prec_leaf=p, prec_mid=p, prec_root=p, nonsymmetric=True, profile=True)


def _exponents(seed, n):
    return np.round(synth.uniform(seed, n, -40.0, 40.0)).astype(int)


# the last one, rows and columns scaled independently, has no power of the pivots that fits it:
# it is factored without the split products
@pytest.mark.parametrize("how,split", [("rows", True), ("columns", True), ("alike", True), ("kinds", True),
                                       ("independently", False)])
@pytest.mark.parametrize("sizes,s_root", [([300, 140], 170), ([600], 90)])
def test_fp64_lu_of_scaled_arrow_fronts(rsd, how, split, sizes, s_root):
    B, owner, parent, kind = _arrow(sizes, s_root, 7000 + sizes[0], how == "kinds")
    n, r0 = len(B), len(B) - s_root
    e1, e2 = _exponents(7100, n), _exponents(7200, n)
    er, ec = {"rows": (e1, 0 * e1), "columns": (0 * e1, e1), "alike": (e1, e1), "kinds": (40 * kind, 40 * kind),
              "independently": (e1, e2)}[how]
    h = _setup(rsd, np.ldexp(B, er[:, None] + ec[None, :]), owner, parent)
    classes = h.profile()
    assert (classes["gemm_tcgen05_f16"]["launches"] > 0, classes["gemm_simt"]["launches"] == 0) == (True, split)
    S = B[r0:, r0:].copy()
    rb, off = np.arange(r0, n), 0
    for c, s in enumerate(sizes):
        i = np.arange(off, off + s)
        L, U = lu_nopivot(B[np.ix_(i, i)])
        X = np.linalg.solve(U.T, B[r0:, off:off + s].T).T
        Y = np.linalg.solve(L, B[off:off + s, r0:])
        rows = np.concatenate([i, rb])
        gl = np.ldexp(h.front_factor(1 + c), er[i][None, :] - er[rows][:, None])
        gu = np.ldexp(h.front_factor_upper(1 + c), -ec[rows][:, None] - er[i][None, :])
        tol = 40 * (s + 1) * 2.2e-16                          # of the unscaled test
        d = np.abs(U).max()
        assert np.abs(gl - np.vstack([L, X])).max() <= tol, c
        assert np.abs(gu - np.vstack([U.T, Y.T])).max() <= tol * d, c
        S -= X @ Y
        off += s
    L, U = lu_nopivot(S)
    tol = 40 * (max(sizes) + s_root) * 2.2e-16
    assert np.abs(np.ldexp(h.front_factor(0), er[rb][None, :] - er[rb][:, None]) - L).max() <= tol
    assert np.abs(np.ldexp(h.front_factor_upper(0), -ec[rb][:, None] - er[rb][None, :]) - U.T).max() <= tol * np.abs(U).max()
    x0 = synth.uniform(7300, n)
    z = h.apply(torch.as_tensor(np.ldexp(B @ x0, er), device="cuda"))
    assert np.abs(np.ldexp(z.cpu().numpy(), ec) - x0).max() <= 1e-12
    h.close()


def test_fp64_lu_of_an_interface_without_a_diagonal(rsd):
    """Interface unknowns with no diagonal entry (constraints): their pivots come from the
    leaf's Schur contribution alone, and nothing of K says what their scale is."""
    B, owner, parent, _ = _arrow([300], 90, 7500, False)
    B[300:, 300:] = 0.0
    h = _setup(rsd, B, owner, parent)
    x0 = synth.uniform(7301, len(B))
    z = h.apply(torch.as_tensor(B @ x0, device="cuda"))
    assert np.abs(z.cpu().numpy() - x0).max() <= 100 * np.linalg.cond(B) * 2.2e-16
    h.close()
