"""Both routes of the spectrum and polarized Raman tails at the edges of their
rules, against the plain float64 definition.

Reference: time-origin averages by numpy's FFT of the zero-padded series and
the cosine transform by numpy's real FFT of the even extension.  Tolerance: a
float64 transform of length N is accurate to a few eps log2(N) of the root
sum of squares, about 1e-15 of the correlation at lag 0; divided by T - tau >=
T / 2 and summed over M lags this stays below 1e-12 of the largest value
(omega^2 weights are relative to the same maximum)."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
REL = 1e-12


@pytest.fixture(scope="module")
def tn():
    from paper_2312_05233_gb300 import tnep
    return tnep


def series(T, C, seed):
    rng = np.random.default_rng(seed)
    t = np.arange(T)[:, None]
    return (rng.standard_normal((1, C)) + 0.1 * np.cos(0.05 * t + rng.uniform(0, 6, (1, C)))
            + 0.05 * rng.standard_normal((T, C)))


def correlate(x, y, M):
    N = 1 << (len(x) + M).bit_length()
    return np.fft.irfft(np.conj(np.fft.rfft(x, N)) * np.fft.rfft(y, N), N)[:M + 1] / (len(x) - np.arange(M + 1))


def cosine(c, dt):
    return dt * np.fft.rfft(np.concatenate([c[:-1], 2 * c[-1:], c[1:-1][::-1]])).real


def close(got, ref):
    np.testing.assert_allclose(got, ref, rtol=0, atol=REL * np.abs(ref).max())


# (T, M): direct below 2e7 terms, segments of 2^7 .. 2^16 samples above, M at,
# below and above a segment's length, lags beyond T / 2, one segment, and the
# cosine transform on both sides of its rule (M = 4000)
SIZES = [(2, 1), (3, 2), (37, 18), (400, 399), (5000, 2500), (60000, 128), (60000, 129), (60001, 127), (30000, 1024),
         (30000, 1023), (30000, 1025), (40000, 3999), (40000, 4000), (40000, 4001), (16384, 8192), (100000, 33000),
         (20000, 12000), (70000, 60000)]


@pytest.mark.parametrize("T,M", SIZES)
@pytest.mark.parametrize("kind", ["ir", "iso", "aniso"])
def test_spectrum_routes(tn, T, M, kind):
    code = {"ir": tn.TNEP_SPECTRUM_IR, "iso": tn.TNEP_SPECTRUM_RAMAN_ISO, "aniso": tn.TNEP_SPECTRUM_RAMAN_ANISO}[kind]
    s = series(T, 3 if kind == "ir" else 9, T + M)
    x = s
    if kind != "ir":
        g = (s[:, 0] + s[:, 4] + s[:, 8])[:, None] / 3
        x = g if kind == "iso" else s - g * np.eye(3).reshape(1, 9)
    x = x - x.mean(0)
    w = x.shape[1]
    pairs = [(c, (c % 3) * 3 + c // 3) for c in range(9)] if kind == "aniso" else [(c, c) for c in range(w)]
    acf = sum(correlate(x[:, p], x[:, q], M) for p, q in pairs) / (3 if kind == "ir" else 1)
    ref = cosine(acf, 0.5)
    nu = np.arange(M + 1) / (2 * M * 0.5)
    if kind == "ir":
        ref = ref * (2 * np.pi * nu) ** 2
    f, S, a = tn.tnep_spectrum(s, 0.5, code, M, want_acf=True)
    if M <= T // 2:
        close(a, acf)
        close(S, ref)
    else:  # few terms per lag at the end: the reference itself is good to eps T / (T - tau)
        np.testing.assert_allclose(a, acf, rtol=0, atol=REL * T / (T - M) * np.abs(acf).max())
        np.testing.assert_allclose(S, ref, rtol=0, atol=REL * T / (T - M) * np.abs(ref).max())
    np.testing.assert_allclose(f, nu / 2.99792458e-5, rtol=1e-14)


@pytest.mark.parametrize("T,M", [(2, 1), (50, 49), (300, 150), (4000, 128), (4001, 129), (9000, 700), (3000, 1500),
                                 (20000, 256), (6000, 4096), (30000, 2048)])
def test_raman_tensor_routes(tn, T, M):
    s = series(T, 9, T * 3 + M)
    x = s - s.mean(0)
    f, L = tn.tnep_raman_tensor(s, 2.0, M)
    slack = 1.0 if M <= T // 2 else T / (T - M)
    ref = np.zeros((M + 1, 9, 9))
    for p in range(9):
        for q in range(p, 9):
            c = 0.5 * (correlate(x[:, p], x[:, q], M) + correlate(x[:, q], x[:, p], M))
            ref[:, p, q] = ref[:, q, p] = cosine(c, 2.0)
    np.testing.assert_allclose(L, ref, rtol=0, atol=slack * REL * np.abs(ref).max())
    np.testing.assert_allclose(f, np.arange(M + 1) / (2 * M * 2.0) / 2.99792458e-5, rtol=1e-14)


@pytest.mark.parametrize("axis", [0, 1, 2])
@pytest.mark.parametrize("n_theta", [1, 16, 17])
def test_porto_map_of_any_tensor(tn, axis, n_theta):
    """The six-coefficient form against the full contraction w L w, for tensors
    that are not symmetric in their pairs; relative to sum |w| |L| |w| the
    rounding is a few eps."""
    rng = np.random.default_rng(axis + 10 * n_theta)
    M = 130
    L = rng.standard_normal((M + 1, 9, 9))
    th = rng.uniform(0, 2 * np.pi, n_theta)
    th[0] = 0.0
    par, crs = tn.tnep_raman_porto_map(L, th, axis=axis)
    a, b = (axis + 1) % 3, (axis + 2) % 3
    e, y = np.zeros((n_theta, 3)), np.zeros((n_theta, 3))
    e[:, a], e[:, b], y[:, a], y[:, b] = np.cos(th), -np.sin(th), np.sin(th), np.cos(th)
    for got, seen in ((par, e), (crs, y)):
        w = (seen[:, :, None] * e[:, None, :]).reshape(n_theta, 9)
        ref = np.einsum("op,kpq,oq->ok", w, L, w)
        size = np.einsum("op,kpq,oq->ok", np.abs(w), np.abs(L), np.abs(w))
        assert np.all(np.abs(got - ref) <= 1e-14 * size.max())
    L[3, axis * 3, 0] = np.nan  # an entry of weight zero
    L[5, a * 3 + a, a * 3 + a] = np.inf
    par, _ = tn.tnep_raman_porto_map(L, th + 0.1, axis=axis)
    assert np.isnan(par[:, 3]).all() and np.isfinite(par[:, 4]).all() and np.isposinf(par[:, 5]).all()


def tensor_reference(x, M, dt):
    """Lineshape tensor of the mean-free x, and a bound on its rounding for each
    component: a lag is good to 4 eps log2(2 M) of sqrt(C_pp(0) C_qq(0)) times
    T / (T - tau) <= 2, and 2 M lags of one sign add up."""
    T = len(x)
    ref = np.zeros((M + 1, 9, 9))
    for p in range(9):
        for q in range(p, 9):
            c = 0.5 * (correlate(x[:, p], x[:, q], M) + correlate(x[:, q], x[:, p], M))
            ref[:, p, q] = ref[:, q, p] = cosine(c, dt)
    size = np.sqrt((x * x).sum(0) / T)
    return ref, 8 * np.finfo(float).eps * np.log2(2 * M) * 2 * M * dt * np.outer(size, size)


# below and above 1e9 terms, one segment and several
@pytest.mark.parametrize("T,M", [(5000, 1000), (3000, 1500), (20000, 3001)])
@pytest.mark.parametrize("sub", [True, False])
@pytest.mark.parametrize("ratio", [1e2, 1e4, 1e8])
def test_small_tensor_components_keep_their_accuracy(tn, T, M, sub, ratio):
    """Diagonal channels `ratio` times the others, a constant one and an empty
    one: the error of every component is relative to its own size."""
    rng = np.random.default_rng(T + M)
    s = rng.standard_normal((T, 9)) + (2.0 if not sub else 300.0)
    s[:, [0, 4, 8]] *= ratio
    s[:, 5] = 7.0
    s[:, 7] = 0.0
    f, L = tn.tnep_raman_tensor(s, 2.0, M, sub)
    x = s - s.mean(0) if sub else s
    if sub:
        x[:, 5] = 0.0
    ref, tol = tensor_reference(x, M, 2.0)
    assert np.all(np.abs(L - ref).max(0) <= tol), np.abs(L - ref).max(0) / tol


@pytest.mark.parametrize("T,M", [(500, 200), (5000, 1000), (20000, 3001)])
@pytest.mark.parametrize("sub", [True, False])
@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_a_channel_that_is_not_finite_spoils_only_its_own_pairs(tn, T, M, sub, bad):
    s = np.random.default_rng(T).standard_normal((T, 9)) + 0.5
    s[T // 3, 1] = bad
    f, L = tn.tnep_raman_tensor(s, 2.0, M, sub)
    s[T // 3, 1] = 0.0
    ref, tol = tensor_reference(s - s.mean(0) if sub else s, M, 2.0)
    mine = np.zeros((9, 9), bool)
    mine[1], mine[:, 1] = True, True
    assert not np.isfinite(L[:, mine]).any()
    assert np.all(np.abs(L - ref).max(0)[~mine] <= tol[~mine])
