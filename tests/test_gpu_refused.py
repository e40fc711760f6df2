"""Axes whose operator would not keep the digit products exact (large steps, long
rows: tc_accept in csrc/sfac_tc_build.cu) stay with the FFT passes: powers of
two, zero-padded, both kinds of axis, and the whole-call launch. Each case first
shows that it runs them: an FFT carries two lines at once, so a line scaled down
by a power of two beside an unscaled one loses bits, where the tensor-core pass
scales every line by itself."""
import numpy as np
import pytest

import paper_2209_08437_gb300 as S
import sfac_inputs as I
from oracle import sfac_oracle as O

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# length: (alpha, eps, tau) on (0, 1); the largest sum is 1.01 to 1.04 of the limit
REFUSED = {255: (1.837, 12.93, 0.002602), 256: (1.399, 6.38, 0.0174), 512: (1.191, 11.1, 0.00527),
           700: (1.638, 2.43, 0.0131), 1024: (1.96, 0.0248, 47.7)}


def problem(n, ax, steps=0):
    al, eps, tau = REFUSED[n[ax]]
    alpha = [1.5] * len(n)
    alpha[ax] = al
    return I.Problem(n=n, alpha=tuple(alpha), eps=eps, tau=tau, a=0.0, b=1.0, steps=steps)


def factor(prob, u, ax):
    """The linear factor of an axis by numpy FFTs on the plan's own eigenvalues:
    these parameters amplify the eigenvalues' rounding (tau times the largest of
    them is 1e3 and more), which is not the pass's."""
    n, d = prob.n[ax], u.ndim
    lam, mu, _, _ = S.sfac.sfac_plan_tables(
        S.sfac.make_params(prob.n, prob.alpha, prob.eps, prob.tau, prob.a, prob.b), ax)
    x = np.moveaxis(u, d - 1 - ax, -1)
    twist = np.exp(1j * np.pi * np.arange(n) / n)
    half = np.exp(0.5 * prob.tau * lam)
    x = np.fft.ifft(half * np.fft.fft(x)).real
    x = (np.fft.ifft(np.exp(prob.tau * mu) * np.fft.fft(x * twist)) * twist.conj()).real
    return np.moveaxis(np.fft.ifft(half * np.fft.fft(x)).real, -1, d - 1 - ax)


def one_pass(prob, u0, ax, jq=(0, 0)):
    with S.Plan.for_problem(prob) as plan:
        u = torch.tensor(np.ascontiguousarray(u0), device="cuda")
        plan.axis_pass(u, ax, *jq)
        plan.check()
        return u.cpu().numpy()


@pytest.mark.parametrize("n,ax", [((255, 20), 0), ((20, 255), 1), ((256, 20), 0), ((20, 256), 1), ((512, 6), 0),
                                  ((6, 512), 1), ((700, 6), 0), ((6, 700), 1), ((1024, 6), 0), ((4, 1024), 1)], ids=str)
def test_fft_passes_of_refused_operators(n, ax):
    prob = problem(n, ax)
    u0 = I.random_field(prob, 87, -1.0, 1.0)
    other = n[1 - ax]
    scale = np.ldexp(1.0, -30 * (np.arange(other) % 2))      # every second line 2^-30
    scale = scale[:, None] if ax == 0 else scale[None, :]
    got = one_pass(prob, u0, ax)
    assert not np.array_equal(got * scale, one_pass(prob, u0 * scale, ax))
    # the rounding of six FFTs on either side, relative to the input, as these
    # factors damp most of it
    assert np.abs(got - factor(prob, u0, ax)).max() <= 2e-14 * np.abs(u0).max()
    flowed = one_pass(prob, u0, ax, (1, 1))
    ref = O.nonlinear_flow(factor(prob, O.nonlinear_flow(u0, 0.5 * prob.tau), ax), 0.5 * prob.tau)
    # the closing flow of 2D 1024 (tau = 47.7) maps small values far apart
    slope = np.exp(0.5 * prob.tau)
    assert np.abs(flowed - ref).max() <= 2e-14 * slope


@pytest.mark.parametrize("n", [(256, 64), (32, 256), (256, 20)], ids=str)
def test_calls_with_a_refused_operator(n):
    """Several steps: one launch for (256, 64) and (32, 256), by FFTs on both axes; one
    pass by FFTs and one on the tensor cores for (256, 20)."""
    prob = problem(n, n.index(256), 4)
    u0 = I.random_field(prob, 88, -0.9, 0.9)
    with S.Plan.for_problem(prob) as plan:
        kind = S.sfac_plan_step_kernel(plan.handle, 4)
        assert kind == (S.sfac.SFAC_STEP_WHOLE if 20 not in n else S.sfac.SFAC_STEP_PASSES)
        u = torch.tensor(u0, device="cuda")
        plan.step(u, 4)
        plan.check()
    ref = u0
    for _ in range(4):
        ref = O.nonlinear_flow(ref, 0.5 * prob.tau)
        for ax in range(2):
            ref = factor(prob, ref, ax)
        ref = O.nonlinear_flow(ref, 0.5 * prob.tau)
    assert np.abs(u.cpu().numpy() - ref).max() <= 1e-13


def test_fp32_refused_operator_takes_the_padded_fft():
    """Entries of 1/2 and more (a large step): the zero-padded FP32 FFT pass. Bar:
    1e-5 in the max norm, as for the other FP32 passes at large steps."""
    prob = I.Problem(n=(100, 40), alpha=(1.5, 1.5), eps=1.0, tau=1.0)
    u0 = I.random_field(prob, 89, -0.9, 0.9).astype(np.float32)
    P = O.Scheme.for_problem(prob).P[0]
    with S.Plan.for_problem(prob, S.SFAC_FP32) as plan:
        u = torch.tensor(u0, device="cuda")
        plan.axis_pass(u, 0, 0, 0)
        plan.check()
    ref = O.apply_axis(u0.astype(np.float64), P, 1)
    assert np.abs(u.double().cpu().numpy() - ref).max() <= 1e-5


# Operators whose sums stay in range row by row, though the largest sums of each
# digit place over all rows, added up, would not: (n, alpha, eps, tau) on (0, 1)
IN_RANGE = [(1024, 1.726, 0.0679, 0.05), (1024, 1.65, 0.0965, 0.05), (1000, 1.838, 7.192, 0.005567),
            (600, 1.636, 0.161, 1.199)]


@pytest.mark.parametrize("n,alpha,eps,tau", IN_RANGE, ids=str)
def test_operators_in_range_are_taken(n, alpha, eps, tau):
    """They run on the tensor cores: lines scale exactly, each by itself."""
    prob = I.Problem(n=(n, 6), alpha=(alpha, 1.5), eps=eps, tau=tau, a=0.0, b=1.0)
    u0 = I.random_field(prob, 92, -1.0, 1.0)
    scale = np.ldexp(1.0, -30 * (np.arange(6) % 2))[:, None]
    got = one_pass(prob, u0, 0)
    assert np.array_equal(got * scale, one_pass(prob, u0 * scale, 0))
    assert np.abs(got - factor(prob, u0, 0)).max() <= 2e-14 * np.abs(u0).max()


@pytest.mark.parametrize("n,ax", [((2048, 6), 0), ((6, 2048), 1), ((4096, 4), 0), ((9, 14), 0), ((14, 9), 1)], ids=str)
@pytest.mark.parametrize("tau", [2e-3, 0.5])
def test_flow_of_the_fft_passes(n, ax, tau):
    """FP64 axes outside 17..1024 points keep the FP64 form of the flow (the probe
    of tests/test_gpu_probe.py runs the fixed-point form): both flows around a
    factor that is the identity to 1e-15. Bar: the rounding of six FFTs and two
    flows of three units each."""
    prob = I.Problem(n=n, alpha=(1.5, 1.5), eps=1e-10, tau=tau)
    u0 = I.random_field(prob, 93, -1.0, 1.0)
    u0.flat[::17] = 0.0
    ref = O.nonlinear_flow(O.nonlinear_flow(u0, 0.5 * tau), tau)
    assert np.abs(one_pass(prob, u0, ax, (1, 2)) - ref).max() <= 2e-14
