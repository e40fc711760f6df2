"""Tensor-core passes at the ends of the field and of the number range."""
import numpy as np
import pytest

import paper_2209_08437_gb300 as S
import sfac_inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,prec", [((33, 1218), S.SFAC_FP64), ((17, 1242), S.SFAC_FP64), ((64, 1300), S.SFAC_FP64),
                                    ((129, 1300), S.SFAC_FP64), ((256, 1218), S.SFAC_FP64), ((65, 70), S.SFAC_FP32),
                                    ((73, 131), S.SFAC_FP32), ((129, 70), S.SFAC_FP32)], ids=str)
@pytest.mark.parametrize("start", [0, 16], ids=["aligned", "mid-sector"])
def test_field_ends_and_mid_sector_starts(n, prec, start):
    """The first and the last lines of a field that begins at a sector or 16 bytes
    into one, with lengths whose last values leave a part of a sector: the bits
    of each line in the middle of a field, and nothing outside is written."""
    dt = torch.float64 if prec == S.SFAC_FP64 else torch.float32
    w, pts = dt.itemsize, n[0] * n[1]
    prob = I.Problem(n=n, alpha=(1.4, 1.6), eps=0.08, tau=0.01)
    u0 = torch.tensor(I.random_field(prob, 83), dtype=dt, device="cuda")
    roll = n[1] // 2
    with S.Plan.for_problem(prob, prec) as plan:
        want = torch.roll(u0, roll, 0).contiguous()      # the ends' lines, in the middle
        plan.axis_pass(want, 0, 1, 0)
        flat = torch.full((pts + 64 // w,), 7.0, dtype=dt, device="cuda")
        lo = start // w
        u = flat[lo:lo + pts].view(u0.shape)
        assert u.data_ptr() % 32 == start
        u.copy_(u0)
        plan.axis_pass(u, 0, 1, 0)
        plan.check()
    assert torch.equal(u, torch.roll(want, -roll, 0))
    assert bool((flat[:lo] == 7.0).all()) and bool((flat[lo + pts:] == 7.0).all())


@pytest.mark.parametrize("n,limit", [((4096, 200), 200_000), ((4096, 300), 300_000), ((4096, 100), 200_000)], ids=str)
def test_limits_do_not_run_during_the_previous_pass(n, limit):
    """A pass may start while the previous one runs (here FP64 FFTs of 4096 points,
    one wave of CTAs of several 100 us that leaves SMs free). The limit of its own
    waits, shorter than that but far above what they take, must not count the
    previous pass: nothing gave up, and the bits are those of the default limit."""
    prob = I.Problem(n=n, alpha=(1.4, 1.6), eps=0.05, tau=1e-3)
    u0 = torch.tensor(I.random_field(prob, 84), device="cuda")
    with S.Plan.for_problem(prob) as plan:
        want = u0.clone()
        plan.step(want, 3)
        plan.check()
        S.sfac_plan_set_wait_limit(plan.handle, limit, 0)
        got = u0.clone()
        plan.step(got, 3)
        plan.check()
    assert torch.equal(got, want)


@pytest.mark.parametrize("n", [(64, 16), (256, 16), (16, 256), (64, 1300), (600, 16), (16, 600)], ids=str)
def test_fp64_lines_near_the_smallest_numbers(n):
    """A line times a power of two gives its result times that power, bit for bit,
    as long as no result is subnormal (2^-900 to 2^-970 at values of 2^-30 and
    more), and within one subnormal unit (2^-1074) of it below."""
    prob = I.Problem(n=n, alpha=(1.4, 1.6), eps=0.1, tau=0.01)
    ax = int(n[1] > n[0] and n[1] < 1000)
    u0 = torch.tensor(I.random_field(prob, 85, -1.0, 1.0), device="cuda")
    with S.Plan.for_problem(prob) as plan:
        want = u0.clone()
        plan.axis_pass(want, ax, 0, 0)
        for k in (-900, -930, -960, -970, -1040):
            got = torch.ldexp(u0, torch.tensor(k / 2, device="cuda"))
            got = torch.ldexp(got, torch.tensor(k / 2, device="cuda"))
            plan.axis_pass(got, ax, 0, 0)
            back = got.cpu().numpy() * 2.0 ** 500 * 2.0 ** (-k - 500)
            w = want.cpu().numpy()
            if k > -1000:
                assert np.array_equal(back, w), k
            else:
                # the field's own rounding (|P| <= 1 in the 2-norm) and the result's
                assert np.abs(back - w).max() <= (np.sqrt(n[ax]) + 1.0) * 2.0 ** (-1075 - k)
        plan.check()


@pytest.mark.parametrize("n", [(100, 40), (40, 100), (255, 33), (33, 255), (127, 9730)], ids=str)
def test_fp32_lines_near_the_smallest_numbers(n):
    """FP32 zero-padded axes: fields of 2^-60 to 2^-125, where the digits' scale has
    no exponent left. Bar: the rounding of y and of the increment (as for fields of
    order one), and the subnormal unit 2^-149 of both."""
    m = (n[0], 70, 139) if n[1] > 1000 else n
    prob = I.Problem(n=m, alpha=(1.3, 1.7, 1.5)[: len(m)], eps=0.05, tau=2e-3)
    ax = 0 if m[0] > 64 else 1
    u0 = torch.tensor(I.random_field(prob, 86, -1.0, 1.0).astype(np.float32), device="cuda")
    with S.Plan.for_problem(prob, S.SFAC_FP32) as plan:
        assert S.sfac_plan_info(plan.handle, ax)[1]
        want = u0.clone()
        plan.axis_pass(want, ax, 0, 0)
        for k in (-60, -90, -100, -108, -112, -120, -125):
            got = u0 * 2.0 ** k
            plan.axis_pass(got, ax, 0, 0)
            back = got.double() * 2.0 ** -k
            # both sides round y and the increment: 6e-8 and 3e-8 at |y| <= 1 each
            assert float((back - want.double()).abs().max()) <= 1.8e-7 + (np.sqrt(m[ax]) + 2.0) * 2.0 ** (-150 - k), k
        plan.check()
