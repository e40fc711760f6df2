"""sfac_diagnostics: both routes against the oracle, and the state it keeps in the plan."""
import threading

import numpy as np
import pytest

import paper_2209_08437_gb300 as S
import sfac_inputs as I
from oracle import sfac_oracle as O

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


@pytest.mark.parametrize("n", [(2048, 3), (8, 1024), (300, 300), (512, 256), (64, 64, 64), (255, 4, 9), (4, 31, 256),
                               (256, 16), (31, 20, 12)], ids=str)
@pytest.mark.parametrize("prec", [S.SFAC_FP64, S.SFAC_FP32])
def test_both_routes_match_oracle(n, prec):
    """Long or many lines take the FFT passes (powers of two, zero-padded, both
    kinds of axis), the last two grids the direct sums. Bar: both parts of the
    energy are positive here, so its relative error is that of the line sums
    (some n roundings, below 1e-12)."""
    prob = I.Problem(n=n, alpha=(1.3, 1.8, 1.5)[: len(n)], eps=0.05, tau=0.01)
    u0 = I.random_field(prob, 15, -1.0, 1.0)
    if prec == S.SFAC_FP32:
        u0 = np.asarray(u0, np.float32).astype(np.float64)
    e_ref = O.discrete_energy(u0, O.Scheme.for_problem(prob, route="spectral"))
    with S.Plan.for_problem(prob, prec) as plan:
        u = torch.tensor(u0, dtype=torch.float64 if prec == S.SFAC_FP64 else torch.float32, device="cuda")
        mx, en = plan.diagnostics(u)
    assert mx == pytest.approx(np.abs(u0).max(), rel=1e-15)
    assert abs(en - e_ref) <= 1e-12 * max(1.0, abs(e_ref)), (en, e_ref)
