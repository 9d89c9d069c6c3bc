"""A block step in two launches (small systems: select, prediction and force in
one kernel) against the same steps made call by call, and its layout (in DS: the
near pairs of HYBRID are chosen from the state, which the step's corrector has
moved on).

Both paths sum the same pair terms; only the order of the double-single partial
sums may differ, each a few 2^-48 of the sum of the terms' magnitudes.  With
cancellation to 1 % of that sum the results agree to ~1e-12 of the largest
value; 1e-10 is asked, far below the FP32 level (6e-8) at which a regrouped FP32
run or a different near pair would show."""
import numpy as np
import pytest

from paper_1104_2700_gb300 import ics

pytestmark = pytest.mark.gpu


def _close(x, y):
    assert np.abs(x - y).max() <= 1e-10 * np.abs(y).max()


@pytest.mark.parametrize("prec", ["hybrid", "ds"])
@pytest.mark.parametrize("n", [2, 33, 64, 65, 129, 1000, 1536, 1537])
def test_block_steps_match_calls(gpu, prec, n):
    m, r, v = ics.plummer(n, 21 + n)
    eps, steps = 4.0 / n, 24
    with gpu.Context(prec) as a, gpu.Context(prec) as b:
        for c in (a, b):
            c.set_particles(m, r, v, eps, 0.02)
        for k in range(steps):
            t, idx = b.select()
            b.predict(t)
            acc, jerk, pot = b.force(idx)
            if k == steps - 1 and prec == "ds":  # a's layout after its step is this prediction
                a.block_step(1.0)
                acc1, jerk1, pot1 = a.force(idx)
                _close(acc1, acc)
                _close(jerk1, jerk)
                _close(pot1, pot)
            else:
                a.block_step(1.0)
            b.correct(t, idx)
        sa, sb = a.get_state(), b.get_state()
    for key in ("r", "v", "a", "j"):
        _close(sa[key], sb[key])
    assert np.array_equal(sa["t"], sb["t"]) and np.array_equal(sa["dt"], sb["dt"])


@pytest.mark.parametrize("prec", ["hybrid", "ds"])
def test_no_block_due(gpu, prec):
    """A step past t_end changes nothing."""
    m, r, v = ics.plummer(300, 5)
    with gpu.Context(prec) as c:
        c.set_particles(m, r, v, 4.0 / 300, 0.02)
        s0 = c.get_state()
        t, _ = c.select()
        c.block_step(t * 0.5)
        s1 = c.get_state()
        assert c.step_until(t * 0.5) == (0, 0)
    for key in s0:
        assert np.array_equal(s0[key], s1[key])


def test_outputs_reorder_between_calls(gpu):
    """The stored order follows the positions at every nb_step_until, also when
    the captured steps serve another end time: a run read at two outputs equals
    one resumed from its own state at the first, bit for bit."""
    n = 700
    m, r, v = ics.plummer(n, 9)
    eps, t1, t2 = 4.0 / n, 2.0 ** -7, 2.0 ** -6
    with gpu.Context("ds", dt_max=2.0 ** -7) as a, gpu.Context("ds", dt_max=2.0 ** -7) as b:
        a.set_particles(m, r, v, eps, 0.02)
        a.step_until(t1)
        s = a.get_state()
        a.step_until(t2)
        b.set_state(m, s["r"], s["v"], s["a"], s["j"], s["t"], s["dt"], eps, 0.02)
        b.step_until(t2)
        sa, sb = a.get_state(), b.get_state()
        assert np.array_equal(a.spatial_order(), b.spatial_order())
    for key in sa:
        assert np.array_equal(sa[key], sb[key])
