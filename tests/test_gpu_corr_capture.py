"""pc_corr under stream capture (after a first call has made its allocations): a replay on
other data leaves the handle as a call would -- the search's matrices, and the product that raw
tests read, which runs on a side stream of the handle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from test_gpu_parity import _random_tests, _sem_case, fp                 # noqa: E402,F401


@pytest.mark.parametrize("p, opts", [(40, {}), (150, {}), (40, dict(order=0)), (40, dict(precision=0))])
def test_replay_equals_call(fp, p, opts):                                # noqa: F811
    Xa, Xb = (torch.from_numpy(_sem_case(s, p, 2000, 0.05)).cuda() for s in (3, 4))
    ij, S = _random_tests(np.random.default_rng(p), p, 1, 500)
    args = torch.from_numpy(ij).cuda(), torch.from_numpy(S).cuda(), 1

    def results(pc):
        return [v.cpu().numpy() for v in pc.ci_batch(*args)] + list(pc.corr_get()) + [pc.skeleton()[0]]
    with fp.PC(2000, p, 0.01, **opts) as pc:
        want = [results(pc.corr(X)) for X in (Xa, Xb)]
    X, s = Xa.clone(), torch.cuda.Stream()
    with fp.PC(2000, p, 0.01, **opts) as pc:
        fp.pc_set_stream(pc.h, s)
        torch.cuda.synchronize()
        pc.corr(X)
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            pc.corr(X)
        for k in (1, 0):
            X.copy_((Xa, Xb)[k])
            torch.cuda.synchronize()
            g.replay()
            torch.cuda.synchronize()
            for a, b in zip(results(pc), want[k]):
                np.testing.assert_array_equal(a, b)
