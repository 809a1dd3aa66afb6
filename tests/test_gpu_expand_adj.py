"""The skeleton as a byte matrix (expand_adj_kernel): 16 entries a thread, for sizes whose rows do
and do not start on a 16-entry boundary, and outputs of any alignment."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from test_gpu_parity import _sem_case, fp                                # noqa: E402,F401


@pytest.mark.parametrize("p", [3, 16, 17, 31, 33, 64, 129, 200])
def test_sizes_and_alignments(fp, p):                                    # noqa: F811
    X = torch.from_numpy(_sem_case(40 + p, p, 600, min(0.9, 6.0 / (p - 1)))).cuda()
    with fp.PC(600, p, 0.01, 1, order=0) as pc:
        pc.corr(X)
        host, _ = pc.skeleton()                          # a host matrix, from the handle's buffer
        removed = set(pc.sepsets())
        want = np.array([[a != b and (min(a, b), max(a, b)) not in removed for b in range(p)] for a in range(p)])
        assert np.array_equal(host.astype(bool), want)
        for off in (0, 1, 4, 7):
            buf = torch.full((p * p + 32,), 9, dtype=torch.uint8, device="cuda")
            out = buf[off:off + p * p].view(p, p)
            pc.skeleton(out)
            got = buf.cpu().numpy()
            assert np.array_equal(got[off:off + p * p].reshape(p, p), host)
            assert (got[:off] == 9).all() and (got[off + p * p:] == 9).all()
