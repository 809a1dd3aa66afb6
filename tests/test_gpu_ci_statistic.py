"""The statistic z of raw CI tests (pc_ci_batch) over the whole range of |r|, up to and
beyond 1, where FP64 decides: every storage of the thread-per-test kernel (registers to 4
members, shared memory to 24) and the warp kernel after it, both precisions, single and
batched handles.

The reference is the definition on the r the call returns: z = sqrt(n-l-3) atanh|r| in
extended precision, infinite from |r| = 1 on.  Tolerances: an FP64-decided z is that value
rounded to FP32 (6e-8) with a function error below 1e-10; an FP32-decided one (its r is an FP32 number) a
few FP32 roundings."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from test_gpu_parity import fp                                           # noqa: E402,F401

LEVELS = [0, 1, 4, 5, 24, 25]


def _pairs(n, p, seed):
    """p columns: the first ones in pairs whose correlation goes from weak to 1 - 1e-16 and exactly 1."""
    rng = np.random.default_rng(seed)
    X = rng.standard_normal((n, p))
    eps = np.r_[3.0, 1.0, 10.0 ** -np.arange(1, 8.5, 0.5), 0.0]
    for k, e in enumerate(eps):
        X[:, 2 * k + 1] = X[:, 2 * k] + e * X[:, 2 * k + 1]
    return X, len(eps)


def _statistic(r, n, l):
    a = np.abs(r.astype(np.longdouble))
    with np.errstate(divide="ignore", invalid="ignore"):
        return np.where(a < 1, np.sqrt(np.longdouble(n - l - 3)) * np.arctanh(a), np.inf).astype(np.float64)


def _tests(pairs, p, l, seed):
    rng = np.random.default_rng(seed)
    ij = np.repeat([[2 * k, 2 * k + 1] for k in range(pairs)], 5, 0).astype(np.int32)
    S = np.stack([rng.choice(np.arange(2 * pairs, p), l, replace=False) for _ in ij]).astype(np.int32).reshape(len(ij), l)
    return ij, S


def _check(r, ind, z, n, l, q):
    want = _statistic(r, n, l)
    f32 = (r == r.astype(np.float32)) & (np.abs(r) < 1)
    for z_, w, tol in ((z[~f32], want[~f32], 8e-8), (z[f32], want[f32], 1e-5)):
        np.testing.assert_array_equal(np.isfinite(z_), np.isfinite(w))
        fin = np.isfinite(w)
        np.testing.assert_allclose(z_[fin], w[fin], rtol=tol, atol=1e-30)
    clear = np.abs(want - q) > 1e-6 * q
    np.testing.assert_array_equal(ind[clear], want[clear] <= q)


@pytest.mark.parametrize("precision", [0, 2])
@pytest.mark.parametrize("l", LEVELS)
def test_statistic_of_strong_pairs(fp, l, precision):                    # noqa: F811
    X, pairs = _pairs(4000, 80, l)
    n, p = X.shape
    ij, S = _tests(pairs, p, l, l + 100)
    with fp.PC(n, p, 0.01, precision=precision) as pc:
        pc.corr(torch.from_numpy(X).cuda())
        r, ind, z = [v.cpu().numpy() for v in pc.ci_batch(torch.from_numpy(ij).cuda(), torch.from_numpy(S).cuda(), l)]
        assert np.abs(r).max() > 1 - 1e-14
        _check(r, ind.astype(bool), z, n, l, fp.pc_threshold(pc.h))


@pytest.mark.parametrize("l", [0, 4, 24])
def test_statistic_in_a_batch(fp, l):                                    # noqa: F811
    Xa, pairs = _pairs(3000, 64, l)
    Xb, _ = _pairs(3000, 70, l + 1)
    ij, S = _tests(pairs, 64, l, l + 100)
    with fp.PCBatch([3000, 3000], [64, 70], 0.01, -1, precision=2) as pb:
        for i, X in enumerate((Xa, Xb)):
            pb.corr_block(i, torch.from_numpy(X).cuda())
        for o in (0, 64):
            r, ind, z = [v.cpu().numpy() for v in pb.ci_batch(torch.from_numpy(ij + o).cuda().int(), torch.from_numpy(S + o).cuda().int(), l)]
            _check(r, ind.astype(bool), z, 3000, l, fp.pc_threshold(pb.h))


@pytest.mark.parametrize("l", [0, 3, 5])
def test_decision_of_duplicates_with_few_samples(fp, l):                 # noqa: F811
    """One degree of freedom and a threshold above the statistic of |r| = 1 - 1e-7: exact duplicates stay dependent."""
    X, pairs = _pairs(l + 4, 48, 7)
    n, p = X.shape
    ij, S = _tests(pairs, p, l, 3)
    for precision in (0, 2):
        with fp.PC(n, p, 1e-25, precision=precision) as pc:
            q = fp.pc_threshold(pc.h)
            assert q > 10.0
            pc.corr(torch.from_numpy(X).cuda())
            r, ind, z = [v.cpu().numpy() for v in pc.ci_batch(torch.from_numpy(ij).cuda(), torch.from_numpy(S).cuda(), l)]
            _check(r, ind.astype(bool), z, n, l, q)
