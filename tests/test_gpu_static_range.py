"""nb_force_static, and NB_DS, in units far from N-body units: the inputs are
doubles, and only what the pair sums need (G m, the positions, the velocities)
has to fit the FP32 pairs they are carried in.  Held to the DS bound, 1e-9 per
particle."""
import ctypes
import os

import numpy as np
import pytest

from paper_1104_2700_gb300 import ics

pytestmark = pytest.mark.gpu
DS_BOUND = 1e-9


def _static(gpu, m, r, v, eps, G, n_act=None):
    torch = pytest.importorskip("torch")
    n = len(m)
    k = n_act or n
    d = [torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (m, r, v)]
    idx = torch.arange(k, dtype=torch.int32, device="cuda")
    out = [torch.empty((k,) + s, dtype=torch.float64, device="cuda") for s in ((3,), (3,), ())]
    torch.cuda.synchronize()
    p = [ctypes.c_void_p(t.data_ptr()) for t in d + [idx] + out]
    assert gpu.nb_force_static(n, *p[:3], eps, G, k, *p[3:], None) == 0
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


@pytest.mark.parametrize("call", ["static", "context"])
@pytest.mark.parametrize("scale", [1e-30, 1e-33, 0.0])
def test_nearly_cold_start(gpu, orc, scale, call):
    """Velocities whose grid quantum has no FP32 reciprocal (largest |v| below
    2^-105 or so).  Their FP32 parts below 2^-126 flush to zero, so each velocity
    is good to 2^-126 of itself and the jerk, against the largest, to a few
    hundred such errors over the largest |v|."""
    n = 1000
    m, r, v = ics.plummer(n, 18)
    v = v * (scale / np.abs(v).max())
    if call == "static":
        acc, jerk, pot = _static(gpu, m, r, v, 4.0 / n, 1.0)
    else:
        with gpu.Context("ds") as c:
            z = np.zeros((n, 3))
            c.set_state(m, r, v, z, z, np.zeros(n), np.full(n, 2.0 ** -10), 4.0 / n, 0.02)
            c.predict(0.0)
            acc, jerk, pot = c.force(np.arange(n, dtype=np.int32))
    a0, j0, p0 = orc.force(m, r, v, 4.0 / n, nthreads=os.cpu_count() or 1)
    assert _err(acc, a0) < DS_BOUND and _err(pot, p0) < DS_BOUND
    assert np.isfinite(jerk).all()
    if scale == 0.0:
        assert not jerk.any()
    else:
        bound = max(DS_BOUND, 300 * 2.0 ** -126 / scale)
        assert np.abs(jerk - j0).max() <= bound * np.abs(j0).max()


@pytest.mark.parametrize("v_scale", [1.0, 1e25])
def test_values_far_from_the_grid(gpu, orc, v_scale):
    """Coordinates far below the grid's quantum beside ordinary ones, and
    velocities above 2^60: the values that are not split on the FP32 pipes."""
    n = 1000
    m, r, v = ics.plummer(n, 19)
    r[::7, 0], r[3::7, 1], r[5::7, 2] = 1e-25, -1e-30, 0.0
    v[::5, 1], v[2::5, 2] = 1e-28, 0.0
    v = v * v_scale
    got = _static(gpu, m, r, v, 4.0 / n, 1.0)
    ref = orc.force(m, r, v, 4.0 / n, nthreads=os.cpu_count() or 1)
    for x, y in zip(got, ref):
        assert _err(x, y) < DS_BOUND


@pytest.mark.parametrize("n_act", [1025, 1500, 1952, 2432])
def test_blocks_above_a_thousand(gpu, orc, n_act):
    """33 to 76 i-groups on this call's grid: equal shares of it or the even
    split, by how the grid divides."""
    n = 3000
    m, r, v = ics.plummer(n, 22)
    got = _static(gpu, m, r, v, 4.0 / n, 1.0, n_act)
    ref = orc.force(m, r, v, 4.0 / n, idx=np.arange(n_act), nthreads=os.cpu_count() or 1)
    for x, y in zip(got, ref):
        assert _err(x, y) < DS_BOUND
