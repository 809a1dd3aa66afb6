"""The error of the FP64 correlations of FP32 data against extended precision, on strongly correlated
columns, whose entries carry the errors of 1/sd whole.  Derived: the two 1/sd 1.5e-16 each (their
double-single sums), the entry about four FP64 roundings of 0.6e-16 (root mean square): 2.5e-16 together,
4e-16 allowed.  A sum that loses the squares of the deviations' low parts is off by 6e-16."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from test_gpu_parity import fp                                           # noqa: E402,F401


@pytest.mark.parametrize("n, mean, scale", [(5000, 0.0, 1.0), (5000, 10.0, 1.0), (20000, 0.0, 1e-6), (20000, 3.0, 1e5)])
def test_error_of_strong_correlations(fp, n, mean, scale):               # noqa: F811
    rng = np.random.default_rng(n + int(mean))
    p = 24
    X = ((rng.standard_normal((n, 1)) + 0.3 * rng.standard_normal((n, p)) + mean) * scale).astype(np.float32)
    L = X.astype(np.longdouble)
    L -= L.mean(0)
    L /= np.sqrt((L * L).sum(0))
    want = L.T @ L
    Xd = torch.from_numpy(X).cuda()
    C = torch.empty((p, p), dtype=torch.float64, device="cuda")
    fp.pc_corr_noalloc(Xd, C)
    torch.cuda.synchronize()
    with fp.PC(n, p, 0.01, precision=0) as pc:
        pc.corr(Xd)
        D = pc.corr_get()[1]
    off = ~np.eye(p, dtype=bool)
    for got in (C.cpu().numpy(), D):
        err = (got.astype(np.longdouble) - want)[off].astype(np.float64)
        assert np.sqrt((err ** 2).mean()) <= 4e-16
