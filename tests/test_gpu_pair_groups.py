"""Stages 1 and 2 by groups of pairs (ci_pairgroup_kernel), whose clearly dependent tests are
decided by a bound: the skeleton, sets and counts of the general kernels, for degrees at the
edges of a group (32 pairs, and fewer once a group's rows fill its shared memory), few samples
(thresholds near 1), singular matrices, wide guards and bands, and batched instances."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2109_04626_gb300 import sem                                   # noqa: E402
from test_gpu_parity import _sem_case, fp                                # noqa: E402,F401

KEYS = ("tests_canonical", "levels_run", "edges_removed", "edges_kept")


def _run(fp, X, pair_warp, **opts):                                      # noqa: F811
    n, p = X.shape
    with fp.PC(n, p, opts.pop("alpha", 0.01), opts.pop("max_level", 2), order=0, stage_loop=0, node_dmax=0,
               pair_warp=pair_warp, pair_warp_dmin=0, **opts) as pc:
        pc.corr(torch.from_numpy(X).cuda())
        adj, st = pc.skeleton()
        return adj, st, pc.sepsets()


def _same(fp, X, **opts):                                                # noqa: F811
    a1, st1, s1 = _run(fp, X, 1, **opts)
    a0, st0, s0 = _run(fp, X, 0, **opts)
    assert np.array_equal(a1, a0) and s1 == s0
    assert all(st1[k] == st0[k] for k in KEYS)


@pytest.mark.parametrize("precision", [1, 2])
@pytest.mark.parametrize("p, n, prob", [(3, 200, 0.9), (33, 4000, 0.9), (34, 4000, 0.9), (65, 5000, 0.8),
                                        (66, 5000, 0.8), (130, 2000, 0.3), (260, 1500, 0.05), (420, 3000, 0.02),
                                        (40, 8, 0.3), (40, 30, 0.6)])
def test_degrees_and_samples(fp, p, n, prob, precision):                 # noqa: F811
    _same(fp, _sem_case(900 + p + n, p, n, prob), precision=precision)


@pytest.mark.parametrize("opts", [dict(guard=0.3), dict(guard=0.0, band=0.5), dict(alpha=0.9), dict(alpha=1e-9),
                                  dict(max_level=1), dict(max_level=-1)])
def test_options(fp, opts):                                              # noqa: F811
    _same(fp, _sem_case(77, 70, 1200, 0.25), **opts)


def test_large_group_rows(fp):                                           # noqa: F811
    """One common cause: every pair stays connected, degrees 511 (24 pairs to a group)."""
    rng = np.random.default_rng(4)
    X = (rng.standard_normal((900, 512)) + 0.8 * rng.standard_normal((900, 1))).astype(np.float32)
    _same(fp, X, max_level=2, budget=1e11)


def test_singular(fp):                                                   # noqa: F811
    X = _sem_case(5, 60, 2000, 0.3)
    X[:, 7] = X[:, 3]
    X[:, 9] = X[:, 3] + 1e-4 * X[:, 9]
    X[:, 11] = 2.5
    _same(fp, X)
    _same(fp, X, precision=1)


def test_batch(fp):                                                      # noqa: F811
    Xs = [_sem_case(30 + i, p, n, pr) for i, (p, n, pr) in enumerate([(50, 40, 0.5), (90, 900, 0.3), (140, 3000, 0.1)])]
    out = []
    for pw in (1, 0):
        with fp.PCBatch([x.shape[0] for x in Xs], [x.shape[1] for x in Xs], 0.01, 2, order=0, node_dmax=0,
                        pair_warp=pw, pair_warp_dmin=0) as pb:
            pb.corr_blocks([torch.from_numpy(x).cuda() for x in Xs])
            adj, st = pb.skeleton(torch.empty((pb.p, pb.p), dtype=torch.uint8, device="cuda"))
            out.append((adj.cpu().numpy(), [st[k] for k in KEYS]))
    assert np.array_equal(out[0][0], out[1][0]) and out[0][1] == out[1][1]


@pytest.mark.parametrize("ps", [(512, 40, 129), (513, 40, 129)])
def test_batch_correlations_at_the_size_limit(fp, ps):                   # noqa: F811
    """Batches of instances of up to 512 variables form every FP64 correlation, larger ones on
    demand: the same matrices (1e-13, and the FP32 rounding or the split product's 1e-6), the
    searches of single handles."""
    import oracle
    Xs = [_sem_case(60 + p, p, 700 + p, 3.0 / p) for p in ps]
    with fp.PCBatch([x.shape[0] for x in Xs], list(ps), 0.01, -1) as pb:
        pb.corr_blocks([torch.from_numpy(x).cuda() for x in Xs])
        adj, st = pb.skeleton()
        adjs, seps = pb.split(adj, pb.sepsets())
        C32, C64 = pb.corr_get()
        o = pb.offsets
    canonical = 0
    for i, X in enumerate(Xs):
        C = oracle.pearson(X)
        np.testing.assert_allclose(C64[o[i]:o[i + 1], o[i]:o[i + 1]], C, rtol=0, atol=1e-13)
        np.testing.assert_allclose(C32[o[i]:o[i + 1], o[i]:o[i + 1]], C, rtol=0, atol=1e-6)
        with fp.PC(*X.shape, 0.01, -1, order=0) as pc:     # a batch runs the conventional order
            pc.corr(torch.from_numpy(X).cuda())
            a, s1 = pc.skeleton()
            assert np.array_equal(a, adjs[i]) and pc.sepsets() == seps[i]
            canonical += s1["tests_canonical"]
    assert canonical == st["tests_canonical"]
