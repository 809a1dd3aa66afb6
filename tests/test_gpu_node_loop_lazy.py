"""FP32 correlations with FP64 entries formed on demand (precision 1, conventional order): the
one-kernel search forms them between its bounded waits, n samples a warp each, so beyond 2^17 samples
the captured loop, which waits for nothing, runs the search."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from test_gpu_parity import _sem_case, fp                                # noqa: E402,F401


@pytest.mark.parametrize("n, order, loop", [(1 << 17, 0, 1), ((1 << 17) + 1, 0, 0), ((1 << 17) + 1, 1, 1)])
def test_samples_limit(fp, n, order, loop):                              # noqa: F811
    X = _sem_case(5, 14, n, 0.3)
    R = oracle.skeleton(oracle.pearson(X), n, 0.01, -1, reversed_order=bool(order))
    with fp.PC(n, 14, 0.01, precision=1, order=order, timing=1) as pc:
        pc.corr(torch.from_numpy(X).cuda())
        adj, st = pc.skeleton()
        np.testing.assert_array_equal(adj, R["adj"])
        assert st["tests_canonical"] == R["tests_total"]
        assert fp.pc_timing(pc.h)["stage_loop"][1] == loop
