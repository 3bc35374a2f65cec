"""ctaux_invert_noalloc on matrices whose rows and columns differ in scale.

The entry point takes any matrix.  Gauss-Jordan elimination with partial
pivoting in float64 is not disturbed by rows of different scale; here its
products run on operands that are rounded relative to the largest element of a
row or column, so the rows of the elimination have to be balanced first.

Rows and columns are scaled by powers of two, so that the exact inverse is that
of the unscaled matrix with the factors taken off again.  The bound is 16 times
the error of the plain float64 elimination of the same matrix, computed here.
"""
import functools

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
pk = pytest.importorskip("paper_1010_3690_gb300")


def _eliminate(a, scaled_pivots):
    """Gauss-Jordan inverse in a's type; pivots by magnitude, or relative to their row."""
    m = len(a)
    w = np.concatenate([a, np.eye(m, dtype=a.dtype)], axis=1)
    for c in range(m):
        mag = np.abs(w[c:, c])
        if scaled_pivots:
            mag = mag / np.abs(w[c:, :m]).max(axis=1)
        p = c + int(np.argmax(mag))
        w[[c, p]] = w[[p, c]]
        w[c] /= w[c, c]
        f = w[:, c].copy()
        f[c] = 0
        w -= f[:, None] * w[c]
    return w[:, m:]


@functools.lru_cache(maxsize=None)
def _base(m, half_column):
    b = np.random.default_rng(m).standard_normal((m, m))
    if half_column:
        b[: m // 2, m - 3] = 0.0
    return b, _eliminate(b.astype(np.longdouble), True)


def _scales(kind, m):
    rng = np.random.default_rng(7 * m + len(kind))
    one = np.ones(m)

    def spread(e):
        return 2.0 ** rng.integers(-e, e + 1, m)

    if kind.startswith("rows"):
        return spread(int(kind[4:])), one
    if kind == "columns":
        return one, spread(53)
    if kind == "both":
        return spread(30), spread(30)
    if kind == "similar":   # D A D^-1, two units
        d = np.where(rng.random(m) < 0.5, 1.0, 2.0 ** 33)
        return d, 1.0 / d
    if kind == "ascending":
        return np.sort(spread(30)), one
    if kind == "half_column":   # a large column that half of the rows do not have
        c = one.copy()
        c[m - 3] = 2.0 ** 27
        return spread(20), c
    near = 2.0 ** rng.integers(-6, 7, m)   # of the smallest and the largest normal number
    end = 2.0 ** (-1010 if kind.startswith("low") else 1005)
    return (near * end, one) if kind.endswith("rows") else (near, one * end)


def _invert(a):
    from paper_1010_3690_gb300 import ctaux
    m = len(a)
    d = torch.tensor(np.ascontiguousarray(a.T), dtype=torch.float64, device="cuda")
    out = torch.full((m, m), float("nan"), dtype=torch.float64, device="cuda")
    logdet = torch.zeros(1, dtype=torch.float64, device="cuda")
    code = ctaux.ctaux_invert_noalloc(d.data_ptr(), m, out.data_ptr(), m, m, logdet.data_ptr(),
                                      torch.cuda.current_stream().cuda_stream)
    assert code == 0
    torch.cuda.synchronize()
    return out.cpu().numpy().T, float(logdet.item())


def _check(m, kind):
    b, exact = _base(m, kind == "half_column")
    r, c = _scales(kind, m)
    a = r[:, None] * b * c[None, :]

    def error(x):
        unscaled = x.astype(np.longdouble) * c[:, None] * r[None, :]
        return float(np.abs(unscaled - exact).max() / np.abs(exact).max())

    inv, logdet = _invert(a)
    plain = max(error(_eliminate(a, False)), m * 2.0 ** -53)
    assert error(inv) <= 16 * plain, (error(inv), plain)
    sign, ref = np.linalg.slogdet(b)
    ref += float(np.sum(np.log(r)) + np.sum(np.log(c)))
    assert logdet == pytest.approx(ref, rel=1e-10, abs=1e-8)


@pytest.mark.parametrize("m", [40, 137, 257])
@pytest.mark.parametrize("kind", ["rows0", "rows13", "rows27", "rows53", "columns", "both", "similar",
                                  "ascending", "half_column", "low", "high",
                                  "low_rows", "high_rows"])
def test_rows_and_columns_of_different_scale(m, kind):
    _check(m, kind)


def test_entry_that_is_not_finite_is_not_lost():
    b, _ = _base(40, False)
    for bad in (np.inf, np.nan):
        a = b.copy()
        a[17, 5] = bad
        inv, logdet = _invert(a)
        assert not np.isfinite(logdet) and (bad == np.inf or np.isnan(inv).any())
