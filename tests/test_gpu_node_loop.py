"""The search of a small problem in one kernel, a CTA per node (csrc/node_loop.cu): the
oracle's skeleton, sets, counts and stages at the edges of its range -- adjacency words of
1 to 4, the smallest p, p at its limit, and every way it hands a stage over to the captured
loop."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle                                                            # noqa: E402
from paper_2109_04626_gb300 import sem                                   # noqa: E402
from test_gpu_parity import _check_skeleton, _run_gpu, _sem_case, fp     # noqa: E402,F401


@pytest.mark.parametrize("order", [0, 1])
@pytest.mark.parametrize("p", [2, 3, 4, 31, 32, 33, 64, 65, 97, 127, 128])
def test_word_edges(fp, p, order):                                       # noqa: F811
    X = _sem_case(700 + p, p, max(200, 12 * p), min(0.9, 5.0 / max(1, p - 1)))
    for precision in (0, 2):
        R, st = _check_skeleton(fp, X, order=order, precision=precision)
        assert st["levels_run"] == len(R["levels"])


@pytest.mark.parametrize("case", ["large_stage", "direct_blocks_off", "deep_stages", "few_samples", "no_closed_form"])
def test_handover_to_the_captured_loop(fp, case):                        # noqa: F811
    if case == "large_stage":            # stage 2 of a dense graph: more sets per node than the kernel takes
        _check_skeleton(fp, sem.make(2).X, order=0)
        _check_skeleton(fp, _sem_case(94, 128, 3000, 0.3), order=0)
    elif case == "direct_blocks_off":    # large sets without precision blocks, from the first stage on
        _check_skeleton(fp, _sem_case(91, 60, 4000, 0.4), order=1, complement=0)
    elif case == "deep_stages":          # dropped sets larger than the complement path's, then stages > 12
        rng = np.random.Generator(np.random.PCG64(613))
        dag, W, o = sem.hub_dag(40, rng, mean_degree=2.0, hubs=2, hub_degree=16, lo=0.4, hi=0.9)
        X = np.ascontiguousarray(sem.sample(W, o, 30000, rng).astype(np.float32))
        _check_skeleton(fp, X, order=0)
        _check_skeleton(fp, X, order=1)
    elif case == "few_samples":          # n near p: FP64 re-decisions, blocks near singular
        for n in (22, 27, 45):
            X = _sem_case(40 + n, 24, n, 0.3)
            _check_skeleton(fp, X, order=0)
            _check_skeleton(fp, X, order=1)
    else:                                # l = p-2 enumerated: one test per ordered pair (the oracle
        X = _sem_case(93, 50, 800, 0.2)  # counts the closed form), so against the captured loop
        a1, st1, s1 = _run_gpu(fp, X, 0.01, -1, 1, 2, stage_a=0)
        a0, st0, s0 = _run_gpu(fp, X, 0.01, -1, 1, 2, stage_a=0, stage_loop=0)
        assert np.array_equal(a1, a0) and s1 == s0
        assert all(st1[k] == st0[k] for k in ("tests_canonical", "levels_run", "first_level", "edges_kept"))


def test_duplicate_and_constant_columns(fp):                             # noqa: F811
    """A singular correlation matrix: no closed-form stage, blocks that fail to build."""
    X = _sem_case(5, 30, 2000, 0.2)
    X[:, 7] = X[:, 3]
    X[:, 11] = 2.5
    _check_skeleton(fp, X, order=1)
    _check_skeleton(fp, X, order=0)


@pytest.mark.parametrize("p, prob, cap", [(2, 1.0, -1), (33, 0.2, -1), (128, 0.04, -1), (64, 0.9, 0), (128, 0.5, 0),
                                          (129, 0.05, -1)])
def test_orient_small_and_dense(fp, p, prob, cap):                       # noqa: F811
    """Phase II in one CTA (p <= 128, mean degree <= 16) and on the whole GPU (denser or
    larger graphs) against the oracle on the same skeleton and sets."""
    X = _sem_case(900 + p, p, 4000, prob)
    with fp.PC(X.shape[0], p, 0.01, cap, order=0) as pc:
        pc.corr(torch.from_numpy(X).cuda())
        adj, _ = pc.skeleton()
        seps = pc.sepsets()
        codes, rounds = pc.orient()
        dev = torch.empty((p, p), dtype=torch.int8, device="cuda")
        pc.orient(dev)
    want, want_rounds = oracle.orient(adj, seps)
    np.testing.assert_array_equal(codes, want)
    np.testing.assert_array_equal(dev.cpu().numpy(), want)
    assert rounds == want_rounds


def test_budget_and_repeated_calls(fp):                                  # noqa: F811
    X = _sem_case(61, 40, 3000, 0.3)
    n, p = X.shape
    with fp.PC(n, p, 0.01, -1, order=0, budget=1000) as pc:
        pc.corr(torch.from_numpy(X).cuda())
        with pytest.raises(fp.PCError) as e:
            pc.skeleton()
        assert e.value.status == 6
        pc.set(budget=1e9)
        a1, _ = pc.skeleton()
        s1 = pc.sepsets()
        a2, _ = pc.skeleton()
        assert np.array_equal(a1, a2) and s1 == pc.sepsets()
