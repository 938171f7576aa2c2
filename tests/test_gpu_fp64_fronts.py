"""FP64 fronts on the GPU: factor, inverted diagonal blocks and Schur contributions of an
arrow matrix (dense leaf blocks, one dense interface) against numpy in FP64, at the edges
of the 32-, 64- and 128-wide blocks and for every cluster size of the diagonal kernel (the
number of fronts picks it)."""
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


def _arrow(sizes, s_root, seed, scale=None):
    """Dense SPD arrow matrix: leaf blocks of the given sizes coupled to s_root interface
    unknowns (the last ones).  Diagonally dominant (condition number below 10), rows and
    columns scaled by `scale` when given."""
    n = sum(sizes) + s_root
    A = np.zeros((n, n))
    owner = np.zeros(n, dtype=np.int32)
    off = 0
    r0 = n - s_root
    for c, s in enumerate(sizes):
        blk = synth.uniform(seed + 2 * c, s * s).reshape(s, s)
        A[off:off + s, off:off + s] = 0.5 * (blk + blk.T)
        cp = synth.uniform(seed + 2 * c + 1, s * s_root).reshape(s, s_root)
        A[off:off + s, r0:] = cp
        A[r0:, off:off + s] = cp.T
        owner[off:off + s] = 1 + c
        off += s
    blk = synth.uniform(seed + 1001, s_root * s_root).reshape(s_root, s_root)
    A[r0:, r0:] = 0.5 * (blk + blk.T)
    A[np.arange(n), np.arange(n)] = 1.25 * (np.abs(A).sum(1) + 1.0)
    if scale is not None:
        A = A * scale[:, None] * scale[None, :]
    parent = np.array([-1] + [0] * len(sizes), dtype=np.int32)
    return A, owner, parent


def _csr(A):
    nz = A != 0.0
    return (torch.as_tensor(np.concatenate([[0], nz.sum(1).cumsum()]).astype(np.int64), device="cuda"),
            torch.as_tensor(np.nonzero(nz)[1].astype(np.int32), device="cuda"),
            torch.as_tensor(A[nz], device="cuda"))


# leaves: 1 front -> 8 CTAs a block, 20 -> 4, 40 -> 2, 80 -> 1 (152 SMs)
@pytest.mark.parametrize("count,edge,s_root", [(1, 1, 3), (1, 33, 129), (2, 128, 31), (3, 130, 200), (2, 600, 90),
                                               (1, 1030, 140), (20, 129, 65), (40, 97, 64), (80, 64, 1), (80, 131, 33)])
def test_fp64_factor_of_arrow_fronts(rsd, count, edge, s_root):
    sizes = [max(1, edge - (c % 3)) for c in range(count)]
    A, owner, parent = _arrow(sizes, s_root, 3000 + 7 * edge)
    p = rsd.RSD_PREC_FP64
    h = rsd.RSD.setup(*_csr(A), torch.as_tensor(owner, device="cuda"), parent, prec_leaf=p, prec_mid=p, prec_root=p)
    n, r0 = A.shape[0], A.shape[0] - s_root
    S = A[r0:, r0:].copy()
    off = 0
    # entries of L and X are at most sqrt(a_ii); FP64 Cholesky of an s-wide block is within
    # (s + 1) eps sqrt(a_ii a_jj) of an exact factor's product, times the condition number
    for c, s in enumerate(sizes):
        blk = A[off:off + s, off:off + s]
        L = np.linalg.cholesky(blk)
        X = np.linalg.solve(L, A[off:off + s, r0:]).T
        got = h.front_factor(1 + c)
        tol = 40 * (s + 1) * 2.2e-16
        d = np.sqrt(np.diag(blk))
        assert (np.abs(got[:s] - L) / d[:, None]).max() <= tol, c
        assert (np.abs(got[s:] - X) / np.sqrt(np.diag(A)[r0:])[:, None]).max() <= tol, c
        for k, D in enumerate(h.front_dinv(1 + c)):
            w = min(128, s - 128 * k)
            Lk = L[128 * k:128 * k + w, 128 * k:128 * k + w]
            assert np.abs(D[:w, :w] @ Lk - np.eye(w)).max() <= tol
            assert not D[w:].any() and not D[:, w:].any() and not np.triu(D, 1).any()
        S -= X @ X.T
        off += s
    got = h.front_factor(0)
    assert (np.abs(got - np.linalg.cholesky(S)) / np.sqrt(np.diag(A)[r0:])[:, None]).max() <= 40 * (max(sizes) + s_root) * 2.2e-16
    f = synth.uniform(4000 + edge, n)
    u, st = h.solve(torch.as_tensor(f, device="cuda"), tol=1e-12)
    assert st["iterations"] == 1
    x = np.linalg.solve(A, f)
    assert np.abs(u.cpu().numpy() - x).max() <= 1e-12 * np.abs(x).max()
    h.close()


@pytest.mark.parametrize("where", ["diag", "below", "coupling"])
@pytest.mark.parametrize("value", [float("nan"), float("inf")])
def test_fp64_front_refuses_values_that_are_not_finite(rsd, where, value):
    A, owner, parent = _arrow([200, 40], 150, 77)
    i, j = {"diag": (3, 3), "below": (190, 5), "coupling": (A.shape[0] - 2, 7)}[where]
    rp, cl, vl = _csr(A)
    row = torch.repeat_interleave(torch.arange(A.shape[0], device="cuda"), rp[1:] - rp[:-1])
    hit = ((row == i) & (cl == j)) | ((row == j) & (cl == i))
    assert int(hit.sum()) == (1 if i == j else 2)
    vl[hit] = value
    p = rsd.RSD_PREC_FP64
    with pytest.raises(rsd.RSDError) as e:
        rsd.RSD.setup(rp, cl, vl, torch.as_tensor(owner, device="cuda"), parent, prec_leaf=p, prec_mid=p, prec_root=p)
    assert e.value.code == -3


def test_fp64_front_refuses_an_indefinite_interface(rsd):
    """A coupling larger than sqrt(a_ii a_jj): every 128-block of the leaf is positive
    definite, the interface is not."""
    A, owner, parent = _arrow([150], 40, 91)
    i, j = A.shape[0] - 3, 11
    A[i, j] = A[j, i] = 50.0 * np.sqrt(A[i, i] * A[j, j])
    p = rsd.RSD_PREC_FP64
    with pytest.raises(rsd.RSDError) as e:
        rsd.RSD.setup(*_csr(A), torch.as_tensor(owner, device="cuda"), parent, prec_leaf=p, prec_mid=p, prec_root=p)
    assert e.value.code == -3


def test_fp64_fronts_of_a_badly_scaled_matrix(rsd):
    """Rows and columns scaled over 2^-40 .. 2^40: the factor's entries scale with them."""
    sizes, s_root = [300, 140], 170
    n = sum(sizes) + s_root
    scale = np.exp2(np.round(synth.uniform(95, n, -40.0, 40.0)))
    A, owner, parent = _arrow(sizes, s_root, 93, scale)
    p = rsd.RSD_PREC_FP64
    h = rsd.RSD.setup(*_csr(A), torch.as_tensor(owner, device="cuda"), parent, prec_leaf=p, prec_mid=p, prec_root=p)
    B, _, _ = _arrow(sizes, s_root, 93)
    L = np.linalg.cholesky(B[:300, :300])
    got = h.front_factor(1)[:300] / scale[:300, None]
    assert (np.abs(got - L) / np.sqrt(np.diag(B)[:300])[:, None]).max() <= 40 * 301 * 2.2e-16
    h.close()


def test_fp64_fronts_in_several_groups_match_one_at_a_time(rsd):
    """Enough leaf rows that the digit workspace holds only part of the level's fronts at
    once (over 10 GB for all): the same applications as each problem alone."""
    n, count = 33, 32
    kinds = [rsd.grid_problem(n, 1, np.exp(synth.normal(500 + q, (n - 1) ** 3)), synth.uniform(600 + q, (n - 2) ** 3))
             for q in range(2)]
    p = rsd.RSD_PREC_FP64
    ref = []
    for k in kinds:
        h = rsd.RSD.setup(k["rowptr"], k["col"], k["val"], k["dof_node"], k["parent"], prec_leaf=p, prec_mid=p, prec_root=p)
        ref.append(h.apply(k["b"]))
        h.close()
    probs = [kinds[(q // 3) % 2] for q in range(count)]
    h = rsd.RSD.setup_batched(probs, prec_leaf=p, prec_mid=p, prec_root=p)
    z = h.apply(torch.cat([q["b"] for q in probs])).reshape(count, -1)
    h.close()
    for q in range(count):
        r = ref[(q // 3) % 2]
        assert float((z[q] - r).abs().max()) <= 1e-13 * float(r.abs().max()), q


@pytest.mark.parametrize("count,edge,s_root", [(1, 1, 3), (1, 33, 129), (2, 128, 31), (3, 130, 200), (2, 600, 90),
                                               (1, 1030, 140), (20, 129, 65), (40, 97, 64), (80, 131, 33)])
def test_fp64_lu_of_arrow_fronts(rsd, count, edge, s_root):
    """Nonsymmetric fronts: L, U, the couplings and L_kk^-1 against LU without pivoting."""
    sizes = [max(1, edge - (c % 3)) for c in range(count)]
    A, owner, parent = _arrow(sizes, s_root, 5000 + 7 * edge)
    skew = synth.uniform(5100 + edge, A.size).reshape(A.shape) * 0.5 * np.abs(A)
    skew[np.arange(len(A)), np.arange(len(A))] = 0.0
    A = A + np.triu(skew, 1) - np.triu(skew, 1).T
    A[np.arange(len(A)), np.arange(len(A))] = 1.25 * (np.abs(A).sum(1) + 1.0)
    p = rsd.RSD_PREC_FP64
    h = rsd.RSD.setup(*_csr(A), torch.as_tensor(owner, device="cuda"), parent, prec_leaf=p, prec_mid=p, prec_root=p,
                      nonsymmetric=True)
    n, r0 = A.shape[0], A.shape[0] - s_root
    S = A[r0:, r0:].copy()
    off = 0
    for c, s in enumerate(sizes):
        L, U = lu_nopivot(A[off:off + s, off:off + s])
        X = np.linalg.solve(U.T, A[r0:, off:off + s].T).T
        Y = np.linalg.solve(L, A[off:off + s, r0:])
        gl, gu = h.front_factor(1 + c), h.front_factor_upper(1 + c)
        tol = 40 * (s + 1) * 2.2e-16                          # (s + 1) eps of each factor's scale, times the condition
        d = np.abs(U).max()
        assert np.abs(gl[:s] - L).max() <= tol and np.abs(gl[s:] - X).max() <= tol, c
        assert np.abs(gu[:s] - U.T).max() <= tol * d and np.abs(gu[s:] - Y.T).max() <= tol * d, c
        for k, D in enumerate(h.front_dinv(1 + c)):
            w = min(128, s - 128 * k)
            assert np.abs(D[:w, :w] @ L[128 * k:128 * k + w, 128 * k:128 * k + w] - np.eye(w)).max() <= tol
            assert not D[w:].any() and not D[:, w:].any() and not np.triu(D, 1).any()
        S -= X @ Y
        off += s
    L, U = lu_nopivot(S)
    tol = 40 * (max(sizes) + s_root) * 2.2e-16
    assert np.abs(h.front_factor(0) - L).max() <= tol
    assert np.abs(h.front_factor_upper(0) - U.T).max() <= tol * np.abs(U).max()
    f = synth.uniform(5200 + edge, n)
    u, st = h.solve(torch.as_tensor(f, device="cuda"), tol=1e-12)
    assert st["iterations"] == 1
    x = np.linalg.solve(A, f)
    assert np.abs(u.cpu().numpy() - x).max() <= 1e-12 * np.abs(x).max()
    h.close()


@pytest.mark.parametrize("where", ["diag", "below", "coupling"])
def test_fp64_lu_front_refuses_values_that_are_not_finite(rsd, where):
    A, owner, parent = _arrow([200, 40], 150, 77)
    i, j = {"diag": (3, 3), "below": (190, 5), "coupling": (A.shape[0] - 2, 7)}[where]
    rp, cl, vl = _csr(A)
    row = torch.repeat_interleave(torch.arange(A.shape[0], device="cuda"), rp[1:] - rp[:-1])
    vl[(row == i) & (cl == j)] = float("nan")
    p = rsd.RSD_PREC_FP64
    with pytest.raises(rsd.RSDError) as e:
        rsd.RSD.setup(rp, cl, vl, torch.as_tensor(owner, device="cuda"), parent, prec_leaf=p, prec_mid=p, prec_root=p,
                      nonsymmetric=True)
    assert e.value.code == -3
