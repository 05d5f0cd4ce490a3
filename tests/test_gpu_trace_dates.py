"""bfm_trace on dates far from 0 (decimal years): the regressors keep FP64 accuracy.

The dates are multiples of 1/64 year and f = 1, so the angles 2 pi j t / f are known
exactly in turns.  The series are the model itself at amplitude 1e6, rounded to float, so
their residuals (about 0.02) show an error of the regressors of 1e-13.  Reference: the
least-squares fit in extended precision.

Tolerance, relative to the amplitude: 2^-44.  The regressors carry 2^-52 and the sums over
180 history dates 180 roundings of 2^-53 if all fall alike (2e-14); the design's
condition number is 3.4.  To that comes the float rounding of the output.  Angles
formed as a product with 2 pi are off by up to 5e-12.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

PI = np.longdouble("3.14159265358979323846264338327950288")


def design(t, k):
    x = [np.ones(len(t), np.longdouble), (t - (t[0] + t[-1]) / 2).astype(np.longdouble) / ((t[-1] - t[0]) / 2)]
    for j in range(1, k + 1):
        a = 2 * PI * (j * t % 1.0).astype(np.longdouble)  # the fraction of a turn is exact
        x += [np.sin(a), np.cos(a)]
    return np.stack(x, 1)


def fit(X, y):
    """Normal equations by Cholesky (numpy's solvers have no extended precision)."""
    K = X.shape[1]
    G, b, L = X.T @ X, X.T @ y, np.zeros((K, K), np.longdouble)
    for i in range(K):
        for j in range(i + 1):
            v = G[i, j] - L[i, :j] @ L[j, :j]
            L[i, j] = np.sqrt(v) if i == j else v / L[j, j]
    for i in range(K):
        b[i] = (b[i] - L[i, :i] @ b[:i]) / L[i, i]
    for i in reversed(range(K)):
        b[i] = (b[i] - L[i + 1:, i] @ b[i + 1:]) / L[i, i]
    return b


@pytest.mark.parametrize("k", [1, 2, 3])
def test_decimal_years(k):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1807_01751_gb300 as bfm
    N, n, m, amp = 300, 180, 16, 1e6
    t = 2000.0 + 3.0 * np.arange(N) / 64.0
    X = design(t, k)
    rng = np.random.default_rng(k)
    coef = rng.uniform(-0.3, 0.3, (X.shape[1], m))
    Y = (amp * (X @ coef)).astype(np.float32)
    Y[rng.random((N, m)) < 0.2] = np.nan
    out = bfm.trace(bfm.Design(t, k, 1.0), torch.from_numpy(Y).cuda(), n_hist=n, h_frac=0.25,
                    status=torch.zeros(m, dtype=torch.uint8, device="cuda"), count=m)
    got = out["resid"].cpu().numpy()
    for p in range(m):
        v = ~np.isnan(Y[:, p])
        y = Y[v, p].astype(np.longdouble)
        hist = np.nonzero(v)[0] < n
        r = y - X[v] @ fit(X[v][hist], y[hist])
        err = np.abs(got[p, v] - r).astype(np.float64)
        assert np.isnan(got[p, ~v]).all()
        assert (err <= 2.0 ** -44 * amp + 2.0 ** -24 * np.abs(r)).all(), (p, err.max() / amp)
