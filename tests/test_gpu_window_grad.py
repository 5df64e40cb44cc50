"""The FP64 adjoint's window operation (both WENO5 states of a five-cell window and their gradients)
through the C ABI (snap_check_weno_grad): in pairs of floats where every difference and indicator
is inside the pairs' range, in FP64 elsewhere.

Windows taken in pairs are compared with the textbook Jiang-Shu formula and its analytic derivative
in extended precision. Bounds: a pair operation is good to u = 2^-46 (products and sums to 2^-47,
a reciprocal from the 23-bit approximation by one correction to 2^-46). A weight carries about
33 u (indicator 6 u, its inverse square 15 u, the normalisation the rest) and a state adds offsets
of at most 2.3 times the window's largest value by weights that sum to one: 33 * 1.4e-14 * 2.3 =
1.1e-12. A gradient entry carries about 90 u on terms that exceed the largest entry by up to ten:
90 * 1.4e-14 * 10 = 1.3e-11. Windows outside the range equal the FP64 form bitwise."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    t = pytest.importorskip("torch")
    if not t.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1901_02955_gb300 import build
    build.build()
    return t


def textbook(X, eps):
    """State at the right face of the middle cell and its gradient, extended precision."""
    L = np.longdouble
    a, b, c, d, e = np.asarray(X, L).T
    n, zero = len(a), np.zeros(len(a), L)
    t = [a - 2 * b + c, b - 2 * c + d, c - 2 * d + e]
    s = [a - 4 * b + 3 * c, b - d, 3 * c - 4 * d + e]
    dt = np.array([[1, -2, 1, 0, 0], [0, 1, -2, 1, 0], [0, 0, 1, -2, 1]], L)
    ds = np.array([[1, -4, 3, 0, 0], [0, 1, 0, -1, 0], [0, 0, 3, -4, 1]], L)
    cand = np.array([[2, -7, 11, 0, 0], [0, -1, 5, 2, 0], [0, 0, 2, 5, -1]], L) / 6
    q = [cand[k] @ np.array([a, b, c, d, e]) for k in range(3)]
    f = [L(eps) + L(13) / 12 * t[k] ** 2 + s[k] ** 2 / 4 for k in range(3)]
    w = [L(m) / f[k] ** 2 for k, m in enumerate((1, 6, 3))]
    S = w[0] + w[1] + w[2]
    w = [x / S for x in w]
    Q = w[0] * q[0] + w[1] * q[1] + w[2] * q[2]
    g = np.zeros((n, 5), L)
    for k in range(3):
        coef = -2 * w[k] * (q[k] - Q) / f[k]
        g += w[k][:, None] * cand[k] + coef[:, None] * (
            L(13) / 6 * t[k][:, None] * dt[k] + s[k][:, None] / 2 * ds[k])
    return Q, g


def run(torch, X, eps, fp64=False):
    from paper_1901_02955_gb300 import capi
    win = torch.tensor(np.ascontiguousarray(X), dtype=torch.float64, device="cuda")
    out = torch.empty((len(X), 13), dtype=torch.float64, device="cuda")
    capi.check_weno_grad(win.data_ptr(), out.data_ptr(), len(X), eps, fp64)
    torch.cuda.synchronize()
    return out.cpu().numpy()


def check_pairs(X, out, eps):
    X, out = X[out[:, 12] == 1.0], out[out[:, 12] == 1.0]
    scale = np.maximum(np.abs(X).max(axis=1), 1e-300)
    for side, Y in ((0, X), (1, X[:, ::-1])):
        Q, g = textbook(Y, eps)
        assert np.all(np.abs(out[:, side] - Q) <= 1.1e-12 * scale)
        err = np.abs(out[:, 2 + 5 * side:7 + 5 * side] - g).max(axis=1)
        assert np.all(err <= 1.3e-11 * np.abs(g).max(axis=1)), float((err / np.abs(g).max(axis=1)).max())


def same(a, b):
    return np.array_equal(a[:, :12], b[:, :12], equal_nan=True)


def test_ordinary_windows(torch):
    rs = np.random.default_rng(21)
    k, m, eps = np.arange(5) - 2.0, 6000, 1e-6
    step = (np.arange(5)[None, :] >= rs.integers(1, 5, size=m)[:, None]).astype(float)
    kinds = [rs.normal(size=(m, 5)),
             rs.normal(size=(m, 1)) + rs.normal(size=(m, 1)) * k + 0.1 * rs.normal(size=(m, 1)) * k ** 2,
             rs.normal(size=(m, 1)) + rs.normal(size=(m, 1)) * step + 1e-3 * rs.normal(size=(m, 5)),
             rs.normal(size=(m, 1)) + rs.normal(size=(m, 1)) * step,
             np.repeat(rs.normal(size=(m, 1)), 5, axis=1),
             1e3 + 1e-2 * rs.normal(size=(m, 5))]
    X = np.concatenate(kinds)
    X = X * rs.choice([1e-3, 1.0, 1e3, 1e5], size=(len(X), 1))
    out = run(torch, X, eps)
    assert np.all(out[:, 12] == 1.0)
    check_pairs(X, out, eps)
    const = np.all(X == X[:, :1], axis=1)
    assert np.array_equal(out[const, 0], X[const, 2]) and np.array_equal(out[const, 1], X[const, 2])


@pytest.mark.parametrize("eps", [1e-6, 1e-30])
def test_every_scale(torch, eps):
    """Random windows of magnitude 10^-30 .. 10^30, smooth and with one value 1e7 times the others:
    the pairs or the FP64 form, whichever the range asks for, and never a wrong result."""
    rs = np.random.default_rng(22)
    m = 400
    X, p = [], []
    for q in range(-30, 31):
        Y = rs.normal(size=(m, 5)) * 10.0 ** q
        Y[: m // 2, :] *= 10.0 ** (7 * (np.arange(5)[None, :] == rs.integers(0, 5, size=m // 2)[:, None]))
        X.append(Y)
        p += [q] * m
    X, p = np.concatenate(X), np.array(p)
    out, ref = run(torch, X, eps), run(torch, X, eps, fp64=True)
    pairs = out[:, 12] == 1.0
    assert not pairs[np.abs(X).max(axis=1) > 1e9].any()
    if eps == 1e-6:
        assert pairs[(p >= -15) & (np.abs(X).max(axis=1) < 1e6)].all()
    else:  # indicators below 1e-15
        assert not pairs[p < -25].any()
    check_pairs(X, out, eps)
    assert same(out[~pairs], ref[~pairs]) and not ref[:, 12].any()


def test_windows_near_rest_stay_in_pairs(torch):
    """Differences below 2^-73 = 1.1e-22 (a field at rest far from what moves) leave the indicators
    and gradients as they are, 1e-22 against sqrt(eps) = 1e-3, but not the states: the same bounds,
    relative to the window's own largest value, for windows of 1e-23 down to the subnormal numbers
    and for windows that mix them with zeros and with larger values at every position."""
    rs = np.random.default_rng(24)
    m, X = 300, []
    for q in (-21, -22, -23, -25, -40, -150, -290, -310):
        Y = rs.normal(size=(m, 5)) * 10.0 ** q
        X += [Y, np.where(rs.random((m, 5)) < 0.4, 0.0, Y),
              np.where(rs.random((m, 5)) < 0.3, rs.normal(size=(m, 5)), Y),
              np.where(rs.random((m, 5)) < 0.3, 1e-18 * rs.normal(size=(m, 5)), Y)]
    X = np.concatenate(X)
    out = run(torch, X, 1e-6)
    assert np.all(out[:, 12] == 1.0)
    check_pairs(X, out, 1e-6)


@pytest.mark.parametrize("jump", [1e8, 1.9e19, 1e20, 1e30])
@pytest.mark.parametrize("step", [False, True])
def test_jumps_beyond_the_range(torch, jump, step):
    """A value (or all values from a position on) so large that the square of a difference leaves
    the floats' range: the FP64 form, to the last bit. Squares overflow from 1.8e19 on."""
    rs = np.random.default_rng(23)
    X = []
    for at in range(5):
        for sign in (-1.0, 1.0):
            Y = rs.normal(size=(200, 5))
            Y[:, at:(5 if step and at else at + 1)] += sign * jump
            X.append(Y)
    X.append(np.array([[jump, 1.3, 1.5, 1.2, 1.1]]))
    X = np.concatenate(X)
    out, ref = run(torch, X, 1e-6), run(torch, X, 1e-6, fp64=True)
    assert not out[:, 12].any()
    assert same(out, ref)


def test_infinite_and_nan_windows_take_the_fp64_form(torch):
    X = np.ones((10, 5))
    X[np.arange(5), np.arange(5)] = np.inf
    X[np.arange(5, 10), np.arange(5)] = np.nan
    out = run(torch, X, 1e-6)
    assert not out[:, 12].any() and same(out, run(torch, X, 1e-6, fp64=True))
    assert not np.isfinite(out[:, 0]).any()


def test_bad_arguments(torch):
    from paper_1901_02955_gb300 import SnapError, capi
    with pytest.raises(SnapError) as e:
        capi.check_weno_grad(0, 0, 2, 1e-6)
    assert e.value.code == capi.EINVAL
    capi.check_weno_grad(0, 0, 0, 1e-6)  # nothing to do
