"""FP32 passes start while the previous one runs and are spread over the SMs by the
shared memory they ask for (launch_spread). Grids whose passes have from a part of a
CTA for every SM to several rounds: a call's steps give the bits of the same passes
launched one at a time with the GPU idle before each."""
import numpy as np
import pytest

import paper_2209_08437_gb300 as S
import sfac_inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [(32, 8), (256, 256), (1024, 256), (512, 100), (64, 128, 64), (32, 32, 512),
                               (256, 256, 64)], ids=str)
def test_same_bits_as_passes_on_an_idle_gpu(n):
    prob = I.Problem(n=n, alpha=(1.4, 1.6, 1.5)[: len(n)], eps=0.06, tau=1e-3)
    u0 = torch.tensor(I.random_field(prob, 82).astype(np.float32))
    d, steps = len(n), 6
    with S.Plan.for_problem(prob, S.SFAC_FP32) as plan:
        a, b = u0.cuda(), u0.cuda()
        for _ in range(steps):
            plan.step(a, 1)
        for _ in range(steps):
            for ax in range(d):
                torch.cuda.synchronize()
                plan.axis_pass(b, ax, int(ax == 0), int(ax == d - 1))
        plan.check()
        assert torch.equal(a, b)
