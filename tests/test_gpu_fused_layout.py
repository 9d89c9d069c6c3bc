"""The j layout that a one-launch block step (HYBRID, small systems) leaves in
global memory, and the same step in HYBRID_SPJ.

The step predicts the tiles in shared memory with the predictor's arithmetic and
stores them, boxes included, so a force call after the step, on the state from
before it, gives the bits of a force call after nb_predict to the same time."""
import numpy as np
import pytest

from paper_1104_2700_gb300 import ics

pytestmark = pytest.mark.gpu
SIZES = [2, 33, 64, 65, 1000, 1536]


@pytest.mark.parametrize("prec", ["hybrid", "hybrid_spj"])
@pytest.mark.parametrize("n", SIZES)
def test_step_leaves_the_predicted_layout(gpu, prec, n):
    torch = pytest.importorskip("torch")
    m, r, v = ics.plummer(n, 31 + n)
    with gpu.Context(prec) as a, gpu.Context(prec) as b:
        for c in (a, b):
            c.set_particles(m, r, v, 4.0 / n, 0.02)
            c.step_until(2.0 ** -8)
        snap = torch.empty(a.snapshot_bytes() // 8 + 1, dtype=torch.float64, device="cuda")
        t, idx = b.select()
        torch.cuda.synchronize()
        a.predict(t + 1.0)  # another layout, to be replaced
        a.snapshot(snap)
        a.block_step(t)
        a.restore(snap)  # a, j, dt and the noise estimates, not the layout
        got = a.force(idx)
        b.predict(t)
        want = b.force(idx)
    for x, y in zip(got, want):
        assert np.array_equal(x, y)


@pytest.mark.parametrize("n", SIZES)
def test_spj_steps_match_calls(gpu, n):
    """The far pairs' jerk is one FP32 sum, grouped differently by the two
    paths: n 2^-24 of the sum of magnitudes at most (1e-4 for 1536), 1e-3 of the
    largest |j|; over steps of 2^-9 at most that is below 1e-6 of r and v.  The
    acceleration's sums stay double-single (and read the states that differ)."""
    m, r, v = ics.plummer(n, 51 + n)
    with gpu.Context("hybrid_spj") as a, gpu.Context("hybrid_spj") as b:
        for c in (a, b):
            c.set_particles(m, r, v, 1.0 / 16, 0.02)
            s = c.get_state()
            c.set_state(m, r, v, s["a"], s["j"], s["t"], np.minimum(s["dt"], 2.0 ** -9),
                        1.0 / 16, 0.02)
        for _ in range(4):
            t, idx = b.select()
            b.predict(t)
            b.force(idx)
            b.correct(t, idx)
            a.block_step(1.0)
        sa, sb = a.get_state(), b.get_state()
    for key, tol in (("r", 1e-6), ("v", 1e-6), ("a", 1e-6), ("j", 1e-3)):
        assert np.abs(sa[key] - sb[key]).max() <= tol * np.abs(sb[key]).max()
