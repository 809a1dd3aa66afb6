"""Executed tests and their flops: every one once, whichever driver ends up with a stage, and none of
the tests that an earlier separation spares."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from test_gpu_parity import _sem_case, fp                                # noqa: E402,F401


def F(l):
    return l ** 3 // 3 + 2 * l * l + 6 * l + 10


def _run(fp, X, cap, **opts):
    with fp.PC(X.shape[0], X.shape[1], 0.01, cap, order=0, **opts) as pc:
        pc.corr(torch.from_numpy(X).cuda())
        return pc.skeleton()


@pytest.mark.parametrize("loop", [0, 1])
def test_stage_handed_over_counts_once(fp, loop):                        # noqa: F811
    """All dependent, and no FP32 test trusted: stage 1 queues more FP64 tests than the one-kernel search
    holds, which hands it over after the FP32 pass.  Every scheduled test is executed exactly once."""
    rng = np.random.default_rng(1)
    p, n = 40, 2000
    X = (rng.standard_normal((n, 1)) + 0.5 * rng.standard_normal((n, p))).astype(np.float32)
    adj, st = _run(fp, X, 1, stage_loop=loop, guard=1e9, pair_warp=0)
    assert adj.sum() == p * (p - 1)
    want = p * (p - 1) + p * (p - 1) * (p - 2)
    assert st["tests_executed"] == st["tests_redecided"] == st["guard_hits"] == want


@pytest.mark.parametrize("p, opts", [(60, {}), (60, dict(stage_loop=0, pair_warp=0)), (60, dict(precision=0))])
def test_flops_of_executed_tests_only(fp, p, opts):                      # noqa: F811
    X = _sem_case(3, p, 2000, 0.15)
    _, st = _run(fp, X, 1, **opts)
    # stage 0 has one test per ordered pair, of which the other side's separation may spare one of two
    e0 = p * (p - 1) // 2, p * (p - 1)
    n, again = st["tests_executed"], st["tests_redecided"]
    assert n > 4 * e0[1]
    assert n * F(1) - e0[1] * (F(1) - F(0)) <= st["flops_class"][3] <= (n + again) * F(1) - e0[0] * (F(1) - F(0))


def test_flops_of_pair_groups(fp):                                       # noqa: F811
    """Tests that the bound decides count their own operations, the others F(1)."""
    X = _sem_case(3, 200, 2000, 0.05)
    _, s0 = _run(fp, X, 0, pair_warp_dmin=0)
    _, s1 = _run(fp, X, 1, pair_warp_dmin=0)
    one = s1["tests_executed"] - s0["tests_executed"]
    got = s1["flops_class"][3] - s0["flops_class"][3]
    assert one > 0 and one * 8 <= got < 0.9 * one * F(1)
