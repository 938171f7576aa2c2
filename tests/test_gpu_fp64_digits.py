"""The digit products of FP64 fronts and the reciprocals of their pivot chains against exact
arithmetic (rationals), on fronts whose every other step is exact."""
from fractions import Fraction

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rsd():
    from paper_1210_6266_gb300 import build
    build.build()
    import paper_1210_6266_gb300 as m
    return m


def _setup(rsd, count, s, diag, low, up, root, nonsymmetric=False):
    """`count` leaves of s unknowns with diagonal blocks diag(diag[c]), leaf c coupled to
    interface unknown c alone (row low[c], column up[c]): every pivot, Schur product and
    interface entry is on its own."""
    n = count * s + count
    rows, cols, vals = [], [], []
    i = np.arange(count * s)
    c = i // s
    for r, q, v in ((i, i, diag), (count * s + c, i, low), (i, count * s + c, up),
                    (count * s + np.arange(count),) * 2 + (root,)):
        rows.append(r)
        cols.append(q)
        vals.append(np.asarray(v, dtype=np.float64).reshape(-1))
    rows, cols, vals = np.concatenate(rows), np.concatenate(cols), np.concatenate(vals)
    o = np.lexsort((cols, rows))
    rowptr = np.concatenate([[0], np.bincount(rows, minlength=n).cumsum()]).astype(np.int64)
    owner = np.concatenate([1 + c, np.zeros(count)]).astype(np.int32)
    p = rsd.RSD_PREC_FP64
    return rsd.RSD.setup(torch.as_tensor(rowptr, device="cuda"), torch.as_tensor(cols[o].astype(np.int32), device="cuda"),
                         torch.as_tensor(vals[o], device="cuda"), torch.as_tensor(owner, device="cuda"),
                         np.array([-1] + [0] * count, dtype=np.int32), prec_leaf=p, prec_mid=p, prec_root=p,
                         nonsymmetric=nonsymmetric)


# s = 512: the longest sum of one update; 130: a block column's update and a ragged last block;
# "flat": entries of like size; "spike": one large entry and small ones, whose squares' left-out
# digits are of one sign (0.27 units at 512 without the diagonal's correction); "graded": over 30 bits
@pytest.mark.parametrize("kind", ["flat", "spike", "graded"])
@pytest.mark.parametrize("s", [130, 512])
def test_schur_products_are_rounded_once(rsd, kind, s):
    """a - sum x^2 with a the sum's FP64 neighbour: all of the leading bits cancel and what is
    left shows the error of the product in units of 2^-53 a.  One rounding is at most half a
    unit (up to 1 where the sum lies just above a power of two), the digit pairs left out
    below 2^-5 of one; the leaf's factor is the identity and the couplings have no bit below the
    59 of a row, so that they come through unchanged."""
    count = 256
    g = np.random.default_rng(11)
    x = g.uniform(0.5, 1.0, (count, s))
    if kind == "spike":
        x[:, 1:] *= 2.0 ** -26
        x[:, 0] = g.uniform(0.5, 0.6, count)
    if kind == "graded":
        x = np.ldexp(x, -g.integers(0, 31, (count, s)))
        x[:, 0] = 0.75
    x = np.ldexp(np.rint(np.ldexp(x, 55)), -55) * g.choice([-1.0, 1.0], (count, s))
    exact = [sum(Fraction(v) ** 2 for v in row) for row in x]
    gap = 2.0 ** -20                                       # keeps every pivot positive
    root = np.array([float(e) + gap for e in exact])
    h = _setup(rsd, count, s, np.ones((count, s)), x, x, root)
    top = h.front_factor(0)
    err = []
    for c in range(count):
        f = h.front_factor(1 + c)
        assert np.array_equal(f[:s], np.eye(s)) and np.array_equal(f[s], x[c])
        want = Fraction(root[c]) - exact[c]
        # (the root's square root is good to 2^-52 of the gap, 2^-20 of a unit's scale)
        err.append(float((Fraction(top[c, c]) ** 2 - want) / Fraction(root[c])) * 2.0 ** 53)
    err = np.array(err)
    print(kind, s, "mean", err.mean(), "max", np.abs(err).max())
    assert np.abs(err).max() <= 1.05
    # uniform over one to two units: the mean of 256 has a deviation of 0.29 / 16 to 0.58 / 16
    assert abs(err.mean()) <= 4 * 0.58 / 16
    h.close()


def _pivots():
    """Mantissas next to 1 and 2, powers of two and between, odd and even exponents, both
    sides of the range in which the chains use their own estimate (2^-1000 .. 2^1000)."""
    g = np.random.default_rng(12)
    m = np.concatenate([[1.0, 1.0 + 2.0 ** -52, 1.0 + 2.0 ** -23, 2.0 - 2.0 ** -52, 2.0 - 2.0 ** -22, 1.5], g.uniform(1.0, 2.0, 26)])
    e = np.concatenate([[-1001, -1000, -999, 999, 1000, 1001, -2, -1, 0, 1, 2], g.integers(-998, 999, 21)])
    return np.ldexp(m[:, None], e[None, :]).reshape(-1)


def test_reciprocal_square_roots_of_pivots(rsd):
    """One-unknown leaves: the inverted block is 1 / sqrt(d), the factor d / sqrt(d).  The estimate is good
    to 2^-21 and the step's remainder to 5/16 e^3 < 2^-61; rounding e gives 2^-54, the result
    2^-53.  Beyond 2^+-1000 a square root and a division, 2^-53 each."""
    d = _pivots()
    count = len(d)
    h = _setup(rsd, count, 1, d, np.zeros(count) + 1e-300, np.zeros(count) + 1e-300, np.full(count, 1.0))
    for c in range(count):
        y = Fraction(float(h.front_dinv(1 + c)[0][0, 0]))
        # y^2 d = 1 + 2 delta + delta^2
        delta = (y * y * Fraction(d[c]) - 1) / 2
        assert abs(delta) <= Fraction(2 if abs(np.log2(d[c])) >= 1000 else 1.52) / 2 ** 53, (d[c], float(delta) * 2 ** 53)
    h.close()


def test_reciprocals_of_pivots(rsd):
    """Two-unknown LU leaves [[d, 0], [1, 1]]: l_21 = 1 / d, up to one rounding (the estimate's error
    is 2^-22, the step leaves its cube)."""
    d = np.concatenate([_pivots(), -_pivots()[::7]])
    count = len(d)
    n = 3 * count
    i = np.arange(count)
    tiny = 1e-300                                          # (the pattern is symmetric)
    a, b, r = 2 * i, 2 * i + 1, 2 * count + i
    rows = np.concatenate([a, b, a, b, r, b, r])
    cols = np.concatenate([a, b, b, a, r, r, b])
    vals = np.concatenate([d, np.ones(count), np.full(count, 0.0), np.ones(count), np.ones(count), np.full(2 * count, tiny)])
    o = np.lexsort((cols, rows))
    rowptr = np.concatenate([[0], np.bincount(rows, minlength=n).cumsum()]).astype(np.int64)
    owner = np.concatenate([1 + np.arange(2 * count) // 2, np.zeros(count)]).astype(np.int32)
    p = rsd.RSD_PREC_FP64
    h = rsd.RSD.setup(torch.as_tensor(rowptr, device="cuda"), torch.as_tensor(cols[o].astype(np.int32), device="cuda"),
                      torch.as_tensor(vals[o], device="cuda"), torch.as_tensor(owner, device="cuda"),
                      np.array([-1] + [0] * count, dtype=np.int32), prec_leaf=p, prec_mid=p, prec_root=p, nonsymmetric=True,
                      profile=True)
    assert h.profile()["gemm_simt"]["launches"] == 0       # (the FP64 pipe's kernel divides)
    for c in range(count):
        y = Fraction(float(h.front_factor(1 + c)[1, 0]))
        delta = y * Fraction(d[c]) - 1
        assert abs(delta) <= Fraction(1.001) / 2 ** 53, (d[c], float(delta) * 2 ** 53)
    h.close()
