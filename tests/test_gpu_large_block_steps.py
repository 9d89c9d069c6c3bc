"""Block steps of every particle at once, above a thousand: one launch serves
blocks of every size in DS, FP64 and the sixth-order scheme, and gives each
i-group an equal share of the CTAs or splits the work evenly over them, as the
grid divides.  Against the same steps made call by call, whose large blocks run
the plain build: the same pair terms in another order, 1e-10 of the largest
value as in the small block steps."""
import numpy as np
import pytest

from paper_1104_2700_gb300 import ics

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["ds", "fp64", "fp64_hermite6"])
@pytest.mark.parametrize("n", [1025, 2016, 2945, 3300])
def test_whole_blocks_match_calls(gpu, prec, n):
    m, r, v = ics.plummer(n, 60 + n)
    with gpu.Context(prec, dt_max=2.0 ** -9) as a, gpu.Context(prec, dt_max=2.0 ** -9) as b:
        a.set_particles(m, r, v, 0.5, 0.02)
        s = a.get_state()
        for c in (a, b):  # all due at once
            c.set_state(m, r, v, s["a"], s["j"], s["t"], np.full(n, 2.0 ** -12), 0.5, 0.02)
        for k in range(3):
            t, idx = b.select()
            assert k > 0 or len(idx) == n
            b.predict(t)
            b.force(idx)
            b.correct(t, idx)
            a.block_step(1.0)
        sa, sb = a.get_state(), b.get_state()
    for key in ("r", "v", "a", "j"):
        assert np.abs(sa[key] - sb[key]).max() <= 1e-10 * np.abs(sb[key]).max()
    assert np.array_equal(sa["t"], sb["t"]) and np.array_equal(sa["dt"], sb["dt"])
