"""FP32 strided passes of 4096 points whose columns come in whole 32-byte sectors run
in clusters that exchange the rows through distributed shared memory
(axis_pass_cluster_rows_kernel). The lines and their arithmetic are those of the
persistent CTA kernel, which a field that starts 16 bytes into a sector, or a
stride that is not a multiple of 8, still takes: same bits."""
import numpy as np
import pytest

import paper_2209_08437_gb300 as S
import sfac_inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [(8, 4096), (24, 2048), (1224, 4096), (16, 4096, 3)], ids=str)
@pytest.mark.parametrize("jq", [(0, 0), (1, 2)], ids=str)
def test_same_bits_as_the_cta_kernel(n, jq):
    prob = I.Problem(n=n, alpha=(1.4, 1.6, 1.5)[: len(n)], eps=0.06, tau=1e-3)
    u0 = I.random_field(prob, 81).astype(np.float32)
    with S.Plan.for_problem(prob, S.SFAC_FP32) as plan:
        flat = torch.zeros(u0.size + 8, dtype=torch.float32, device="cuda")
        a, b = flat[:u0.size].view(u0.shape), None
        assert a.data_ptr() % 32 == 0
        a.copy_(torch.tensor(u0))
        plan.axis_pass(a, 1, *jq)
        got = a.cpu().numpy()
        b = flat[4:4 + u0.size].view(u0.shape)          # 16 bytes into a sector
        b.copy_(torch.tensor(u0))
        plan.axis_pass(b, 1, *jq)
        plan.check()
        assert np.array_equal(got, b.cpu().numpy())
