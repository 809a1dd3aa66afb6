"""Stages above l = 12 by a warp per test (ci_direct_kernel), whose matrix of up to 16 or 24 rows is
factored in registers: the oracle's skeleton, sets and counts with the other small-stage layouts
off."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2109_04626_gb300 import sem                                   # noqa: E402
from test_gpu_parity import _check_skeleton, fp                          # noqa: E402,F401


@pytest.mark.parametrize("precision", [1, 2])
@pytest.mark.parametrize("degree", [14, 15, 16, 19])
def test_hub_stages(fp, degree, precision):                              # noqa: F811
    """One hub that keeps its neighbours: stages up to l = degree - 1, few tests in the last ones."""
    rng = np.random.Generator(np.random.PCG64(degree))
    p, n = degree + 6, 20000
    Z = rng.standard_normal((n, p))
    Z[:, 0] += 0.5 * Z[:, 1:degree + 1].sum(1)
    X = np.ascontiguousarray(Z.astype(np.float32))
    R, st = _check_skeleton(fp, X, order=0, precision=precision, stage_loop=0, node_dmax=0, pair_warp=0)
    assert st["levels_run"] == len(R["levels"])
