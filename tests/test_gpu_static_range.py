"""nb_force_static in units far from N-body units: its inputs are doubles, and
only what the pair sums need (G m, the positions, the velocities) has to fit the
FP32 pairs they are carried in.  Held to the DS bound, 1e-9 per particle."""
import ctypes
import os

import numpy as np
import pytest

from paper_1104_2700_gb300 import ics

pytestmark = pytest.mark.gpu
DS_BOUND = 1e-9


def _static(gpu, m, r, v, eps, G):
    torch = pytest.importorskip("torch")
    n = len(m)
    d = [torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (m, r, v)]
    idx = torch.arange(n, dtype=torch.int32, device="cuda")
    out = [torch.empty((n,) + s, dtype=torch.float64, device="cuda") for s in ((3,), (3,), ())]
    torch.cuda.synchronize()
    p = [ctypes.c_void_p(t.data_ptr()) for t in d + [idx] + out]
    assert gpu.nb_force_static(n, *p[:3], eps, G, n, *p[3:], None) == 0
    return [x.cpu().numpy() for x in out]


def _err(x, ref):
    x, ref = x.reshape(len(x), -1), ref.reshape(len(ref), -1)
    return (np.linalg.norm(x - ref, axis=1) / np.linalg.norm(ref, axis=1)).max()


@pytest.mark.parametrize("G,scale", [(6.674e-8, 1e42), (6.674e-8, 1e40), (1e30, 1e-42),
                                     (0.0043009, 1e6), (1.0, 1.0)])
def test_masses_that_only_g_brings_into_range(gpu, orc, G, scale):
    """m beyond a float's range (a total of 1e42 g, cgs) or below it, with G m
    well inside."""
    n = 1000
    m, r, v = ics.plummer(n, 17)
    m = m * scale
    got = _static(gpu, m, r, v, 4.0 / n, G)
    ref = orc.force(m, r, v, 4.0 / n, G=G, nthreads=os.cpu_count() or 1)
    for x, y in zip(got, ref):
        assert np.isfinite(x).all() and _err(x, y) < DS_BOUND
