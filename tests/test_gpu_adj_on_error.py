"""A device skeleton output stays as it was when pc_skeleton fails, whichever driver ran the stages
before the error: the one-kernel search, its hand-over to the captured loop, and the captured
or the host loop alone."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from test_gpu_parity import _sem_case, fp                                # noqa: E402,F401


@pytest.mark.parametrize("p, opts", [(40, {}), (40, dict(order=0)), (40, dict(order=0, graph=0)), (40, dict(order=0, stage_loop=0)),
                                     (150, dict(order=0)), (150, dict(order=0, graph=0))])
def test_output_untouched_on_a_budget_error(fp, p, opts):                # noqa: F811
    X = torch.from_numpy(_sem_case(50 + p, p, 1500, 10.0 / p)).cuda()
    with fp.PC(1500, p, 0.01, **opts) as pc:
        pc.corr(X)
        want, st = pc.skeleton()
        out = torch.full((p, p), 9, dtype=torch.uint8, device="cuda")
        # at the first stage; after some (conventional order: stage 0 has p (p - 1) tests)
        for budget in (1.0, 2.0 * p * p) if "order" in opts else (1.0,):
            pc.set(budget=budget)
            with pytest.raises(fp.PCError) as e:
                pc.skeleton(out)
            assert e.value.status == 6
            assert (out == 9).all()
        pc.set(budget=2e10)
        pc.skeleton(out)
        np.testing.assert_array_equal(out.cpu().numpy(), want)
