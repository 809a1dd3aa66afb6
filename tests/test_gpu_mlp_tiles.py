"""The proposal network's forward and gradient kernels at the edges of their tiles (128 rows),
of their groups (a chain per group, several per CTA) and on unaligned rows, against FP64
arithmetic on the same BF16-rounded operands.

Tolerance 1e-3 of a result's norm: FP32 accumulation (2^-24 a term) shifts a few values across
a BF16 rounding boundary (2^-8 of one of at least 128 terms each); a wrong tile, row or
column is off by a whole term."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from test_gpu_parity import fp                                           # noqa: E402,F401


def _bf(x):
    return x.to(torch.bfloat16).double()


def _reference(theta, F, y):
    w1, b1, w2, b2, w3, b3 = torch.from_numpy(theta).cuda().split([2048, 128, 16384, 128, 128, 1])
    x, W1, W2 = _bf(F), _bf(w1.view(128, 16)), _bf(w2.view(128, 128))
    b1, b2, w3, b3 = b1.double(), b2.double(), w3.double(), b3.double()
    h1 = _bf(torch.relu(x @ W1.T + b1).float())
    h2 = torch.relu(h1 @ W2.T + b2)
    s = h2 @ w3 + b3
    ds = (torch.sigmoid(s) - y.double()) / len(s)
    da2 = _bf((ds[:, None] * w3 * (h2 > 0)).float())
    da1 = _bf(((da2 @ W2) * (h1 > 0)).float())
    g = torch.cat([(da1.T @ x).reshape(-1), da1.sum(0), (da2.T @ h1).reshape(-1), da2.sum(0), h2.T @ ds, ds.sum()[None]])
    loss = torch.nn.functional.binary_cross_entropy_with_logits(s, y.double())
    return s, g, float(loss)


def _off(a, b):
    return float((a.double() - b).norm() / b.norm())


@pytest.mark.parametrize("R", [1, 2, 127, 128, 129, 255, 256, 257, 600, 152 * 128 - 1, 152 * 128 + 1, 304 * 128 + 5,
                               608 * 128, 608 * 128 + 1, 100001])
@pytest.mark.parametrize("shift", [0, 1])
def test_tiles(fp, R, shift):                                            # noqa: F811
    rng = np.random.default_rng(R)
    theta = (rng.standard_normal(fp.pc_mlp_nparam()) * 0.15).astype(np.float32)
    buf = torch.from_numpy(rng.uniform(-1, 1, R * 16 + shift).astype(np.float32)).cuda()
    F = buf[shift:].view(R, 16)                           # shift 1: rows off the 16-byte boundary
    y = torch.from_numpy((rng.random(R) < 0.4).astype(np.float32)).cuda()
    s, g, loss = _reference(theta, F, y)
    with fp.PC(100, 10, 0.01) as pc:
        fp.pc_mlp_set_params(pc.h, theta)
        assert _off(fp.pc_mlp_forward(pc.h, F), s) < 1e-3
        got, l = fp.pc_mlp_grad(pc.h, F, y)
        assert abs(l - loss) < 1e-5 * (1 + loss)
        got = torch.from_numpy(got).cuda()
        o = 0
        for size in (2048, 128, 16384, 128, 128, 1):      # every block of parameters by itself
            assert _off(got[o:o + size], g[o:o + size]) < 1e-3, (o, size)
            o += size
        again, l2 = fp.pc_mlp_grad(pc.h, F, y)            # fixed order of every sum
        assert np.array_equal(again, got.cpu().numpy()) and l2 == l
        fp.pc_set_opt(pc.h, "mlp_backward", 0)            # FP32 backward from saved activations
        ref, l3 = fp.pc_mlp_grad(pc.h, F, y)
        assert _off(torch.from_numpy(ref).cuda(), g) < 2e-2 and abs(l3 - loss) < 1e-5 * (1 + loss)
