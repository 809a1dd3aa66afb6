"""The FP64 correlation matrix by exact integer products on the tensor cores
(csrc/gram_exact.cu) through pc_corr_noalloc, at the edges of its tiles (128 x 48, 32
samples per stage, 512 samples per split), unaligned rows, large means, scales far from 1,
heavy tails, constant columns and non-finite input.

Tolerance on a correlation, against sums in extended precision: the fixed-point rounding
of x and the dropped digit weights 2^-54 each, four FP64 roundings of the result 2^-51, and
the two standard deviations (double-single or FP64 sums) 1e-15 relative each: 4e-15."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from test_gpu_parity import fp                                           # noqa: E402,F401

TOL = 4e-15


def _want(X):
    X = X.astype(np.longdouble)
    D = X - X.mean(0)
    sd = np.sqrt((D * D).sum(0))
    with np.errstate(divide="ignore", invalid="ignore"):
        D = np.where(sd > 0, D / sd, 0)
    # accumulate in extended precision without its (slow) matrix product
    C = np.zeros((X.shape[1],) * 2, dtype=np.longdouble)
    for a in range(X.shape[1]):
        C[a] = (D * D[:, a:a + 1]).sum(0)
    np.fill_diagonal(C, 1)
    return C.astype(np.float64)


def _run(fp, X, pad=0):
    n, p = X.shape
    big = torch.full((n, p + pad), 7.0, dtype=torch.from_numpy(X).dtype, device="cuda")
    big[:, :p] = torch.from_numpy(X).cuda()
    C = torch.full((p, p + 3), 5.0, dtype=torch.float64, device="cuda")
    fp.pc_corr_noalloc(big[:, :p], C[:, :p])
    assert bool((C[:, p:] == 5.0).all())
    return C[:, :p].cpu().numpy()


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("p, n, pad", [(1, 40, 0), (2, 2, 0), (7, 33, 1), (31, 600, 0), (47, 31, 2), (48, 32, 0),
                                       (49, 513, 3), (96, 1000, 0), (127, 64, 1), (128, 511, 0), (129, 512, 5),
                                       (130, 1537, 0), (257, 300, 0)])
def test_tile_edges(fp, p, n, pad, dtype):                               # noqa: F811
    rng = np.random.default_rng(p * 1000 + n)
    X = (rng.standard_normal((n, p)) @ (np.eye(p) + 0.2 * rng.standard_normal((p, p)))).astype(dtype)
    np.testing.assert_allclose(_run(fp, X, pad), _want(X), rtol=0, atol=TOL)


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("case", ["means", "scales", "tails", "constant"])
def test_values(fp, case, dtype):                                        # noqa: F811
    rng = np.random.default_rng(11)
    n, p = 3000, 60
    X = rng.standard_normal((n, p)) @ (np.eye(p) + 0.3 * rng.standard_normal((p, p)))
    tol = TOL
    if case == "means":
        X += 10.0 ** rng.integers(0, 4, p)
        # the mean's own rounding, 2^-53 |mean| / sd, enters at second order only
    elif case == "scales":
        X *= 10.0 ** rng.integers(-12, 12, p)
    elif case == "tails":
        X = np.sign(X) * np.abs(X) ** 5                  # the largest deviations near sqrt(n) sd
        X[17, 3] = 1e6
    else:
        X[:, 5] = 3.25
        X[:, 20] = 0.0
        X[:, 21] = X[:, 22]
    X = X.astype(dtype)
    np.testing.assert_allclose(_run(fp, X), _want(X), rtol=0, atol=tol)


def test_non_finite_columns(fp):                                         # noqa: F811
    rng = np.random.default_rng(3)
    X = rng.standard_normal((500, 20)).astype(np.float32)
    Y = X.copy()
    X[9, 4], X[11, 13] = np.nan, np.inf
    C, W = _run(fp, X), _want(Y)
    bad = np.zeros(20, bool)
    bad[[4, 13]] = True
    off = ~np.eye(20, dtype=bool)
    assert np.isnan(C[bad][:, ~bad]).all() and np.isnan(C[~bad][:, bad]).all()
    assert (np.diag(C) == 1.0).all()
    good = np.outer(~bad, ~bad) & off
    np.testing.assert_allclose(C[good], W[good], rtol=0, atol=TOL)


def test_repeatable(fp):                                                 # noqa: F811
    X = np.random.default_rng(5).standard_normal((5000, 200)).astype(np.float32)
    assert np.array_equal(_run(fp, X), _run(fp, X))      # integer accumulation: any order, the same bits


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
def test_fixed_point_limits(fp, dtype):                                  # noqa: F811
    """FP32 input: columns on both sides of the limits of the 32-bit fixed point (|mean| against
    8 sqrt(n) sd, 2^s a normal FP32 number), next to each other in a group of 8 columns."""
    rng = np.random.default_rng(17)
    n, p = 500, 40
    X = rng.standard_normal((n, p)) @ (np.eye(p) + 0.3 * rng.standard_normal((p, p)))
    sd = X.std(0)
    X += np.sqrt(n) * sd * np.where(np.arange(p) < 16, 2.0 ** (np.arange(p) % 16 - 8), 0.0)
    X[:, 16:24] += np.sqrt(n) * sd[16:24] * np.array([3.9, 4.1, 7.9, 8.1, -3.9, -4.1, -7.9, -8.1])
    X[:, 24:32] *= 10.0 ** np.array([-32, -28, -24, -20, 20, 25, 30, 34])
    X = X.astype(dtype)
    np.testing.assert_allclose(_run(fp, X), _want(X), rtol=0, atol=TOL)
