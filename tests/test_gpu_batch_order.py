"""A batched handle's instances may be given in any order, on device memory that holds
anything, and one at a time again: the matrices are bit for bit those of the ascending
order, and the skeletons are found."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from test_gpu_batch import _instances, fp                                # noqa: E402,F401


def _leave_dirty_memory():
    """Give back device memory whose every word is non-zero, in blocks of several sizes."""
    for words in (1 << 8, 1 << 16, 1 << 19, 1 << 23):
        blocks = [torch.full((words,), 7, dtype=torch.int32, device="cuda") for _ in range(32)]
        torch.cuda.synchronize()
        del blocks
        torch.cuda.empty_cache()


@pytest.mark.parametrize("precision", [0, 2])
@pytest.mark.parametrize("order", [(4, 3, 2, 1, 0), (2, 4, 0, 1, 3)])
def test_instances_in_any_order(fp, precision, order):                   # noqa: F811
    inst = _instances(5, 930, p_range=(20, 70), n_range=(400, 2000))
    ns, ps = [s.X.shape[0] for s in inst], [s.X.shape[1] for s in inst]
    Xs = [torch.from_numpy(s.X).cuda() for s in inst]
    got = []
    for seq in (range(5), order):
        for _ in range(3):
            with fp.PCBatch([900] * 3, [11, 140, 33], 0.01, -1):
                pass
            _leave_dirty_memory()
            with fp.PCBatch(ns, ps, 0.01, -1, precision=precision) as pb:
                for i in seq:
                    pb.corr_block(i, Xs[i])
                C32, C64 = pb.corr_get()
                adj, st = pb.skeleton()
                pb.corr_block(order[0], Xs[order[0]])    # one of them again
                D32, D64 = pb.corr_get()
            assert np.isfinite(C64).all() and np.isfinite(C32).all()
            np.testing.assert_array_equal(C64, D64)
            np.testing.assert_array_equal(C32, D32)
            got.append((C32, C64, adj, st["tests_canonical"]))
    for g in got[1:]:
        for a, b in zip(got[0], g):
            np.testing.assert_array_equal(a, b)
