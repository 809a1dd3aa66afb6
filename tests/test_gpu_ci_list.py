"""Raw CI tests (pc_ci_batch), a thread per test: every set size at the edges of its two
storages (registers to 4 members, shared memory to 24, 128 or 64 threads) and of the warp
kernel after it, odd batch sizes, invalid ids beside valid ones, degenerate sets -- against
the FP64 oracle, and bit for bit against the warp kernel where FP32 decides.

Tolerances: an FP32-decided r carries the error bound 5e-6 (set size <= 3); an FP64-decided
one the conditioning of its set times a few FP64 roundings, far below 1e-9 here."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle                                                            # noqa: E402
from test_gpu_parity import _random_tests, _sem_case, fp                 # noqa: E402,F401


def _batch(pc, ij, S, l):
    r, ind, z = pc.ci_batch(torch.from_numpy(ij).cuda(), torch.from_numpy(S).cuda(), l)
    return r.cpu().numpy(), ind.cpu().numpy().astype(bool), z.cpu().numpy()


@pytest.mark.parametrize("l, b", [(0, 1), (0, 1000), (1, 129), (2, 5000), (3, 127), (4, 128), (5, 333), (15, 65),
                                  (16, 129), (17, 64), (24, 1), (24, 500), (25, 40), (60, 9)])
@pytest.mark.parametrize("precision", [0, 2])
def test_sizes(fp, l, b, precision):                                     # noqa: F811
    X = _sem_case(31, 150, 3000, 0.04)
    n, p = X.shape
    C = oracle.pearson(X)
    ij, S = _random_tests(np.random.default_rng(l * 7 + b), p, l, b)
    ro, zo, io, do = oracle.ci_batch(C, n, 0.01, ij, S)
    with fp.PC(n, p, 0.01, precision=precision) as pc:
        pc.corr(torch.from_numpy(X).cuda())
        r, ind, z = _batch(pc, ij, S, l)
        st = fp.pc_last_stats(pc.h)
    assert np.abs(r - ro).max() <= (1e-9 if precision == 0 or l >= 4 else 5e-6)
    clear = np.abs(zo - oracle.threshold(0.01)) > 1e-9
    np.testing.assert_array_equal(ind[clear], io[clear])
    assert st["tests_executed"] == b
    if precision == 2:
        with fp.PC(n, p, 0.01, order=0) as pc:           # FP64 entries on demand: the warp kernel
            pc.corr(torch.from_numpy(X).cuda())
            rw, iw, zw = _batch(pc, ij, S, l)
            sw = fp.pc_last_stats(pc.h)
        f32 = rw == rw.astype(np.float32)                # decided in FP32 (an FP64 value is no float)
        np.testing.assert_array_equal(r[f32], rw[f32])
        np.testing.assert_array_equal(z[f32], zw[f32])
        assert np.abs(r - rw).max() <= 1e-9
        np.testing.assert_array_equal(ind, iw)
        assert all(st[k] == sw[k] for k in ("tests_redecided", "band_hits", "guard_hits", "degenerate"))


@pytest.mark.parametrize("l", [1, 2, 6, 20])
def test_degenerate_and_strong(fp, l):                                   # noqa: F811
    """Duplicate and nearly duplicate columns (pivots at the floor, |r| near 1)."""
    X = _sem_case(8, 140, 2000, 0.05)
    rng = np.random.default_rng(l)
    X[:, 1] = X[:, 0]
    X[:, 3] = X[:, 2] + (1e-3 * rng.standard_normal(len(X))).astype(np.float32)
    n, p = X.shape
    C = oracle.pearson(X)
    ij, S = _random_tests(rng, p, l, 400)
    S[:100, 0], ij[:100] = 0, [[1, 7]]
    ij[100:200] = [[2, 3]]
    for t in range(200):                                  # sets without the pair's nodes
        pool = np.setdiff1d(np.arange(4, p), np.r_[ij[t]])
        S[t, 1 if t < 100 else 0:] = rng.choice(pool, l - (t < 100), replace=False)
    ro, zo, io, do = oracle.ci_batch(C, n, 0.01, ij, S)
    with fp.PC(n, p, 0.01) as pc:
        pc.corr(torch.from_numpy(X).cuda())
        r, ind, z = _batch(pc, ij, S, l)
    assert np.abs(r - ro).max() <= 1e-5
    clear = np.abs(zo - oracle.threshold(0.01)) > 1e-6
    np.testing.assert_array_equal(ind[clear], io[clear])


def test_invalid_ids(fp):                                                # noqa: F811
    X = _sem_case(9, 40, 500, 0.1)
    n, p = X.shape
    with fp.PC(n, p, 0.01) as pc:
        pc.corr(torch.from_numpy(X).cuda())
        for l in (0, 2, 9):
            ij, S = _random_tests(np.random.default_rng(l), p, l, 300)
            for bad in ([0, 0], [-1, 3], [2, p]):
                q = ij.copy()
                q[17] = bad
                with pytest.raises(fp.PCError) as e:
                    _batch(pc, q, S, l)
                assert e.value.status == 1
            _batch(pc, ij, S, l)
