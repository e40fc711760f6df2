"""FP64 passes of 17..1024 points on the tensor cores (csrc/sfac_tc_*.cu):
the edges of their tiles (lengths around the folding limit 128, the K step 32,
the cluster limits 256, 512 and 768, odd lengths, line counts around the tile
widths 8..64), the scaling of each line, non-finite values, and the bounded
wait."""
import numpy as np
import pytest

import paper_2209_08437_gb300 as S
import sfac_inputs as I
from oracle import sfac_oracle as O

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# Rounding of y (1.1e-16), digits below order 9 and the fixed-point rounding of x
# (together below 5e-16), and the dense oracle factor's own rounding at n = 256
# (5e-15, pinned in test_oracle_pins.py).
TOL = 6e-15


def passes(prob, u0, jq=(0, 0)):
    out = []
    with S.Plan.for_problem(prob) as plan:
        for ax in range(prob.dim):
            u = torch.tensor(np.ascontiguousarray(u0), device="cuda")
            plan.axis_pass(u, ax, *jq)
            plan.check()
            out.append(u.cpu().numpy())
    return out


@pytest.mark.parametrize("n", [(17, 31), (32, 33), (63, 64), (65, 96), (127, 128), (129, 130), (255, 256), (7, 256), (256, 9),
                               (160, 200), (32, 8, 33), (129, 3, 5)], ids=str)
def test_lengths_around_the_tile_edges(n):
    prob = I.Problem(n=n, alpha=(1.2, 1.8, 1.5)[: len(n)], eps=0.08, tau=0.01)
    u0 = I.random_field(prob, 71, -1.0, 1.0)
    sch = O.Scheme.for_problem(prob)
    for ax, got in enumerate(passes(prob, u0)):
        ref = O.apply_axis(u0, sch.P[ax], ax + 1)
        assert np.abs(got - ref).max() <= TOL * np.abs(ref).max(), ax


@pytest.mark.parametrize("n", [(64, 13, 187), (48, 5, 973), (256, 3, 811), (33, 23, 423), (130, 10, 973)], ids=str)
def test_tile_widths(n):
    """Line counts around 16, 32 and 64 times the device's 152 SMs: tiles of 16
    lines (2431), 32 (2433) and 64 (4865; 9729 and 9730: a second round), with a
    partly filled last tile; the contiguous axis and the last one."""
    for m, ax in ((n, 0), ((n[1], n[2], n[0]), 2)):
        prob = I.Problem(n=m, alpha=(1.3, 1.7, 1.5), eps=0.08, tau=0.01)
        u0 = I.random_field(prob, 72, -1.0, 1.0)
        P = O.Scheme.for_problem(I.Problem(n=(n[0],), alpha=(prob.alpha[ax],), eps=0.08, tau=0.01)).P[0]
        with S.Plan.for_problem(prob) as plan:
            u = torch.tensor(np.ascontiguousarray(u0), device="cuda")
            plan.axis_pass(u, ax, 0, 0)
            plan.check()
        ref = O.apply_axis(u0, P, ax + 1)
        assert np.abs(u.cpu().numpy() - ref).max() <= TOL * np.abs(ref).max()


@pytest.mark.parametrize("n", [(257, 33), (33, 258), (300, 31), (511, 3), (512, 32), (16, 513), (769, 9), (1023, 2),
                               (40, 1024), (3, 1000, 11)], ids=str)
def test_long_lines(n):
    """257..1024 points: a cluster of 2, 3 or 4 CTAs per tile of 32 lines (partly
    filled row blocks, 32-column steps and tiles). Reference: the spectral route
    (1.1e-15 per application at n = 1024, pinned in test_oracle_pins.py) plus the
    pass's own 6e-16."""
    prob = I.Problem(n=n, alpha=(1.3, 1.7, 1.5)[: len(n)], eps=0.05, tau=1e-3)
    u0 = I.random_field(prob, 76, -1.0, 1.0)
    ax = int(np.argmax(n))
    one = I.Problem(n=(n[ax],), alpha=(prob.alpha[ax],), eps=0.05, tau=1e-3)
    sch = O.Scheme.for_problem(one)
    got = passes(prob, u0)[ax]
    lines = np.moveaxis(u0, len(n) - 1 - ax, -1).reshape(-1, n[ax])
    ref = np.stack([O.apply_axis(v, sch.P[0], 1) for v in lines[:: max(1, len(lines) // 7)]])
    mine = np.moveaxis(got, len(n) - 1 - ax, -1).reshape(-1, n[ax])[:: max(1, len(lines) // 7)]
    # (the dense factor's rounding at n = 1024: 1.5e-14, pinned likewise)
    assert np.abs(mine - ref).max() <= 2e-14 * np.abs(ref).max()
    if jq_matters(prob):
        u = torch.tensor(np.ascontiguousarray(u0), device="cuda")
        with S.Plan.for_problem(prob) as plan:
            plan.axis_pass(u, ax, 1, 2)
            plan.check()
        flowed = O.nonlinear_flow(ref_all(u0, sch, ax, len(n), 0.5 * prob.tau), prob.tau)
        assert np.abs(u.cpu().numpy() - flowed).max() <= 2e-14 * np.abs(flowed).max()


def jq_matters(prob):
    return prob.points <= 40000


def ref_all(u0, sch, ax, dim, s):
    v = np.moveaxis(O.nonlinear_flow(u0, s), dim - 1 - ax, -1)
    shape = v.shape
    out = np.stack([O.apply_axis(w, sch.P[0], 1) for w in v.reshape(-1, shape[-1])]).reshape(shape)
    return np.moveaxis(out, -1, dim - 1 - ax)


@pytest.mark.parametrize("n", [(64, 16), (256, 16), (16, 256), (600, 16), (16, 600)], ids=str)
def test_lines_scale_exactly(n):
    """A line times a power of two gives its result times that power, bit for
    bit: each line is scaled by its own largest value."""
    prob = I.Problem(n=n, alpha=(1.4, 1.6), eps=0.1, tau=0.01)
    ax = int(np.argmax(n))
    u0 = I.random_field(prob, 73, -1.0, 1.0)
    k = np.arange(16) * 25 - 200                                   # 2^-200 .. 2^175
    scale = np.ldexp(1.0, k)
    scale = scale[:, None] if ax == 0 else scale[None, :]
    a, b = passes(prob, u0)[ax], passes(prob, u0 * scale)[ax]
    assert np.array_equal(a * scale, b)


def test_zero_and_non_finite_lines():
    prob = I.Problem(n=(256, 16), alpha=(1.4, 1.6), eps=0.1, tau=0.01)
    u0 = I.random_field(prob, 74, -1.0, 1.0)
    want = passes(prob, u0)[0]
    u0[3] = 0.0
    u0[5, 17] = np.inf
    u0[9, 200] = np.nan
    got = passes(prob, u0)[0]
    assert np.array_equal(got[3], np.zeros(256))
    assert np.isnan(got[5]).all() and np.isnan(got[9]).all()
    rest = [i for i in range(16) if i not in (3, 5, 9)]
    assert np.array_equal(got[rest], want[rest])


def test_non_finite_long_lines():
    prob = I.Problem(n=(600, 40), alpha=(1.4, 1.6), eps=0.1, tau=0.01)
    u0 = I.random_field(prob, 77, -1.0, 1.0)
    want = passes(prob, u0, (1, 1))[0]
    u0[3] = 0.0
    u0[5, 17] = np.inf
    u0[39, 400] = np.nan
    got = passes(prob, u0, (1, 1))[0]
    assert np.array_equal(got[3], np.zeros(600))
    assert np.isnan(got[5]).all() and np.isnan(got[39]).all()
    rest = [i for i in range(40) if i not in (3, 5, 39)]
    assert np.array_equal(got[rest], want[rest])


@pytest.mark.parametrize("n", [(256, 96), (64, 96), (600, 96), (64, 3000 // 2)], ids=str)
def test_wait_runs_out_and_the_plan_stays_usable(n):
    prob = I.Problem(n=n, alpha=(1.4, 1.6), eps=0.1, tau=1e-2)
    u0 = I.random_field(prob, 75)
    with S.Plan.for_problem(prob) as plan:
        u = torch.tensor(u0, device="cuda")
        S.sfac_plan_set_wait_limit(plan.handle, 100_000, 1)
        plan.axis_pass(u, 0, 0, 0)
        with pytest.raises(S.SfacError) as ei:
            plan.check()
        assert ei.value.status == S.sfac.SFAC_ETIMEOUT
        plan.check()                                  # the flag was cleared
        S.sfac_plan_set_wait_limit(plan.handle, 1 << 32, 0)
        a = torch.tensor(u0, device="cuda")
        plan.axis_pass(a, 0, 1, 2)
        plan.check()
    assert np.array_equal(a.cpu().numpy(), passes(prob, u0, (1, 2))[0])


@pytest.mark.parametrize("n", [(65, 70), (100, 4866), (127, 9730), (129, 66), (255, 2433), (255, 9730), (200, 130)], ids=str)
def test_fp32_padded_lengths(n):
    """FP32 zero-padded axes of 65..256 points: tiles of 16, 32 and 64 lines, odd lines that start at every 4-byte offset, both
    kinds of axis, with and without the flow. Bar: the rounding of y (6e-8 at
    |y| <= 1), the increment (3e-8) and the flow's increments (2 x 3e-8)."""
    m = n[1] // 14 if n[1] > 256 else n[1]
    rest = (m, n[1] // m) if n[1] > 256 else (m,)
    for shape, ax in (((n[0],) + rest, 0), (rest + (n[0],), len(rest))):
        prob = I.Problem(n=shape, alpha=(1.3, 1.7, 1.5)[: len(shape)], eps=0.05, tau=2e-3)
        u0 = I.random_field(prob, 78, -1.0, 1.0).astype(np.float32)
        P = O.Scheme.for_problem(I.Problem(n=(n[0],), alpha=(prob.alpha[ax],), eps=0.05, tau=2e-3)).P[0]
        with S.Plan.for_problem(prob, S.SFAC_FP32) as plan:
            assert S.sfac_plan_info(plan.handle, ax)[1]          # zero-padded
            for jq in ((0, 0), (1, 2)):
                u = torch.tensor(np.ascontiguousarray(u0), device="cuda")
                plan.axis_pass(u, ax, *jq)
                plan.check()
                ref = u0.astype(np.float64)
                ref = O.nonlinear_flow(ref, 0.5 * prob.tau) if jq[0] else ref
                ref = O.apply_axis(ref, P, ax + 1)
                ref = O.nonlinear_flow(ref, prob.tau) if jq[1] else ref
                assert np.abs(u.double().cpu().numpy() - ref).max() <= 1.8e-7


ROUTES = [((255, 63), S.SFAC_FP64), ((300, 40), S.SFAC_FP64), ((128, 96, 100), S.SFAC_FP64), ((127, 250), S.SFAC_FP32),
          ((1024, 64), S.SFAC_FP32), ((32, 256, 80), S.SFAC_FP32), ((16, 2048), S.SFAC_FP32)]


def field(prob, prec, seed):
    dt = torch.float64 if prec == S.SFAC_FP64 else torch.float32
    return torch.tensor(np.ascontiguousarray(I.random_field(prob, seed)), dtype=dt, device="cuda")


@pytest.mark.parametrize("n,prec", ROUTES, ids=str)
def test_steps_in_a_cuda_graph(n, prec):
    """The overlapped launches of a call's passes can be captured and replayed:
    same bits as the direct calls."""
    prob = I.Problem(n=n, alpha=(1.3, 1.7, 1.5)[: len(n)], eps=0.06, tau=2e-3)
    with S.Plan.for_problem(prob, prec) as plan:
        u, ref = field(prob, prec, 79), field(prob, prec, 79)
        for _ in range(3):
            plan.step(ref, 1)
        torch.cuda.synchronize()
        side = torch.cuda.Stream()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.stream(side):
            with torch.cuda.graph(g, stream=side):
                plan.step(u, 1, stream=side.cuda_stream)
        u.copy_(field(prob, prec, 79))
        for _ in range(3):
            g.replay()
        torch.cuda.synchronize()
        plan.check()
    assert torch.equal(u, ref)


@pytest.mark.parametrize("n,prec", ROUTES, ids=str)
def test_one_plan_on_two_streams(n, prec):
    """The passes keep nothing in the plan: two fields advance on two streams at
    the same time with the bits of one after the other."""
    prob = I.Problem(n=n, alpha=(1.3, 1.7, 1.5)[: len(n)], eps=0.06, tau=2e-3)
    with S.Plan.for_problem(prob, prec) as plan:
        want = [field(prob, prec, 90 + i) for i in range(2)]
        for u in want:
            for _ in range(6):
                plan.step(u, 1)
        got = [field(prob, prec, 90 + i) for i in range(2)]
        torch.cuda.synchronize()
        streams = [torch.cuda.Stream() for _ in range(2)]
        for _ in range(6):
            for u, s in zip(got, streams):
                plan.step(u, 1, stream=s.cuda_stream)
        torch.cuda.synchronize()
        plan.check()
    assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])
