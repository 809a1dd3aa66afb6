"""Phase II of graphs with very large degrees: the work between two barriers of the cooperative
kernel could outlast their bound there, so every phase is a launch of its own; one step
below the limit it is one kernel.  Both against the oracle's Phase II on the same sets."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from test_gpu_parity import fp                                           # noqa: E402,F401


def _near_complete(p, holes, seed, n=3000):
    """Variables of one common factor, all dependent but `holes` disjoint pairs that are independent of
    each other alone (x_i = f + g, x_j = f - g): l = 0 removes these only."""
    rng = np.random.default_rng(seed)
    f = rng.standard_normal((n, 1))
    X = f + 0.5 * rng.standard_normal((n, p))
    idx = rng.permutation(p)[:2 * holes].reshape(-1, 2)
    g = rng.standard_normal((n, holes))
    X[:, idx[:, 0]] = f + g
    X[:, idx[:, 1]] = f - g
    return X.astype(np.float32)


def _with_a_chain(p, seed, n=3000):
    """The same without holes, and beside it five variables a -> c <- b, c -> d -> e: a collider, then R1 twice."""
    rng = np.random.default_rng(seed)
    X = rng.standard_normal((n, 1)) + 0.5 * rng.standard_normal((n, p))
    i = rng.permutation(p)[:5]
    a, b, c, d, e = rng.standard_normal((5, n))
    c += a + b
    d += c
    X[:, i] = np.stack([a, b, c, d, d + e], 1)
    return X.astype(np.float32)


@pytest.mark.parametrize("p, holes, phases", [(900, 5, False), (1100, 0, True), (1100, 7, True), (900, None, False),
                                              (1100, None, True)])
def test_dense_graph(fp, p, holes, phases):                              # noqa: F811
    X = _with_a_chain(p, p) if holes is None else _near_complete(p, holes, p + holes)
    with fp.PC(X.shape[0], p, 1e-6, 1 if holes is None else 0, order=0) as pc:
        pc.corr(torch.from_numpy(X).cuda())
        adj, st = pc.skeleton()
        assert st["edges_kept"] >= (p - 5) * (p - 6) // 2
        out = torch.empty((p, p), dtype=torch.int8, device="cuda")
        before = fp.pc_kernel_launches()
        _, rounds = pc.orient(out)
        launches = fp.pc_kernel_launches() - before
        ref, ref_rounds = oracle.orient(adj, pc.sepsets())
    np.testing.assert_array_equal(out.cpu().numpy(), ref)
    assert rounds == ref_rounds
    assert rounds == (2 if holes is None else 0)
    assert launches == (4 + 2 * rounds if phases else 1)


def test_batch_of_dense_graphs(fp):                                      # noqa: F811
    """The limit counts an instance's own words, not those of the batch: a kernel for small instances."""
    Xs = [_near_complete(120, 3, s, 1000) for s in range(40)]
    with fp.PCBatch([1000] * 40, [120] * 40, 1e-6, 0) as pb:
        pb.corr_blocks([torch.from_numpy(X).cuda() for X in Xs])
        adj, _ = pb.skeleton()
        adjs, seps = pb.split(adj, pb.sepsets())
        before = fp.pc_kernel_launches()
        codes, _ = pb.orient()
        assert fp.pc_kernel_launches() - before == 1
    for i, (a, s) in enumerate(zip(adjs, seps)):
        o = 120 * i
        np.testing.assert_array_equal(codes[o:o + 120, o:o + 120], oracle.orient(a, s)[0])
