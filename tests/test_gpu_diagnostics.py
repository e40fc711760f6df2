"""sfac_diagnostics: the state it keeps in the plan."""
import threading

import pytest

import paper_2209_08437_gb300 as S
import sfac_inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [(64, 64), (127, 127), (1024, 256)], ids=str)
def test_calls_after_overlapping_ones_are_right(n):
    """Two threads that call sfac_diagnostics on one plan at once share its scratch
    and may spoil each other's values, but no later call's: the arrival counter
    is 0 again once they have finished."""
    prob = I.Problem(n=n, alpha=(1.3, 1.7), eps=0.05, tau=0.01)
    fields = [torch.tensor(I.random_field(prob, 17 + i), device="cuda") for i in range(2)]
    with S.Plan.for_problem(prob) as plan:
        want = [plan.diagnostics(u) for u in fields]
        start = threading.Barrier(2)

        def many(u):
            stream = torch.cuda.Stream()
            start.wait()
            for _ in range(100):
                plan.diagnostics(u, stream=stream.cuda_stream)

        for _ in range(5):
            threads = [threading.Thread(target=many, args=(u,)) for u in fields]
            for t in threads:
                t.start()
            for t in threads:
                t.join()
            torch.cuda.synchronize()
            assert [plan.diagnostics(u) for u in fields] == want
