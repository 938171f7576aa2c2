"""TF32 fronts on the GPU: factor and inverted diagonal blocks of an arrow matrix (dense
leaf blocks, one dense interface) against numpy in FP64, at the edges of the 128-wide
blocks and of the 512-wide panels, with one and several fronts on a level."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from test_gpu_fp64_fronts import _arrow, _csr, rsd  # noqa: E402,F401


# columns [0, 128), [0, 512): one block, one panel; 513 and above: the panels look ahead
@pytest.mark.parametrize("count,edge,s_root", [(1, 1, 3), (1, 127, 130), (3, 129, 5), (1, 383, 513), (2, 512, 140),
                                               (1, 513, 641), (2, 642, 70), (1, 1030, 1100), (20, 140, 260)])
def test_tf32_factor_of_arrow_fronts(rsd, count, edge, s_root):  # noqa: F811
    sizes = [max(1, edge - (c % 3)) for c in range(count)]
    A, owner, parent = _arrow(sizes, s_root, 7000 + 7 * edge)
    p = rsd.RSD_PREC_TF32
    h = rsd.RSD.setup(*_csr(A), torch.as_tensor(owner, device="cuda"), parent, prec_leaf=p, prec_mid=p, prec_root=p)
    n, r0 = A.shape[0], A.shape[0] - s_root

    def bound(M, L, s):
        # L = (M - L L^T) Linv^T with operands rounded by at most u = 2^-11 of themselves: two
        # operands of each update, M and Linv, what Linv's own products carry (three
        # roundings, through |Linv| |L| |Linv|), and the stored entry.
        u = 2.0 ** -11
        Li, La = np.abs(np.linalg.inv(L[:s])), np.abs(L)
        P = La @ La[:s].T
        return u * ((2 * P + 2 * (np.abs(M) + P)) @ Li.T + 3 * (np.abs(M) + P) @ (Li @ La[:s] @ Li).T + La)

    def check(got, L, tol, c):
        lo = np.tril(np.ones(L.shape, dtype=bool))
        assert (np.abs(got - L) <= tol)[lo].all(), (c, (np.abs(got - L) / tol)[lo].max())

    S = A[r0:, r0:].copy()
    dS = np.zeros_like(S)
    off = 0
    for c, s in enumerate(sizes):
        blk = A[off:off + s, off:off + s]
        L = np.linalg.cholesky(blk)
        X = np.linalg.solve(L, A[off:off + s, r0:]).T
        got = np.asarray(h.front_factor(1 + c))
        tol = bound(np.concatenate([blk, A[r0:, off:off + s]]), np.concatenate([L, X]), s)
        check(got, np.concatenate([L, X]), tol, c)
        tx, ax = tol[s:], np.abs(X)
        dS += tx @ ax.T + ax @ tx.T + 2 * 2.0 ** -11 * ax @ ax.T
        for k, D in enumerate(h.front_dinv(1 + c)):
            w = min(128, s - 128 * k)
            Lk = np.tril(got[128 * k:128 * k + w, 128 * k:128 * k + w])
            # D and L are each rounded once
            tol = 2 * 2.0 ** -11 * np.abs(D[:w, :w]) @ np.abs(Lk) + 1e-5
            assert (np.abs(D[:w, :w] @ Lk - np.eye(w)) <= tol).all()
            assert not D[w:].any() and not D[:, w:].any() and not np.triu(D, 1).any()
        S -= X @ X.T
        off += s
    got = np.asarray(h.front_factor(0))
    L = np.linalg.cholesky(S)
    Li = np.abs(np.linalg.inv(L))
    # the leaves' Schur products change the root by dS, its factor by at most L (Linv dS Linv^T)
    check(got, L, bound(S, L, s_root) + np.abs(L) @ (Li @ dS @ Li.T), "root")
    f = synth.uniform(8000 + edge, n)
    u, st = h.solve(torch.as_tensor(f, device="cuda"), tol=1e-12)
    x = np.linalg.solve(A, f)
    # condition number below 10
    assert np.abs(u.cpu().numpy() - x).max() <= 1e-11 * np.abs(x).max() and st["iterations"] <= 6
    h.close()
