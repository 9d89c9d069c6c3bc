"""Tiles cut between warps whose particles have the integration guard on, and a
device list that names particles twice, in two i-groups of one launch.

In HYBRID the evaluation of the first group stores noise estimates that the
second group's warps may or may not see when they choose between the far and the
near path of a tile, and a tile may be cut between several warps.  Whatever each
warp sees, every record of a tile counts once: the choice may change a term's
precision, never the sum, so both rows of a particle stay within the precision's
1e-6 of the oracle.  (A lost eighth of one of the 128 tiles shows as ~1e-3.)

The state is loaded without noise estimates and with steps so short that the
first evaluation switches every particle's guard on; a second context's large
force call on another stream keeps some of the list's CTAs waiting."""
import os

import numpy as np
import pytest

from paper_1104_2700_gb300 import ics

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows", [33, 64, 200])
def test_particles_named_twice(gpu, orc, rows):
    torch = pytest.importorskip("torch")
    n, eps, repeats = 8192, 4.0 / 8192, 100
    m, r, v = ics.plummer(n, 12)
    nt = os.cpu_count() or 1
    a, j, _ = orc.force(m, r, v, eps, nthreads=nt)
    once = np.sort(ics.permutation(n, 8)[:32]).astype(np.int32)
    lst = np.resize(once, rows)
    _, _, p0 = orc.force(m, r, v, eps, idx=once, nthreads=nt)
    ref = [np.resize(x, (rows,) + x.shape[1:]) for x in (a[once], j[once], p0)]
    side, main = torch.cuda.Stream(), torch.cuda.Stream()
    with gpu.Context("hybrid", stream=main) as c, gpu.Context("hybrid", stream=side) as other:
        dt = np.full(n, 2.0 ** -30)
        c.set_state(m, r, v, a, j, np.zeros(n), dt, eps, 0.02)
        other.set_state(m, r, v, a, j, np.zeros(n), dt, eps, 0.02)
        other.predict(0.0)
        idx = torch.from_numpy(lst).cuda()
        every = torch.arange(n, dtype=torch.int32, device="cuda")
        out = [torch.empty((repeats, rows) + s, dtype=torch.float64, device="cuda")
               for s in ((3,), (3,), ())]
        big = [torch.empty((n,) + s, dtype=torch.float64, device="cuda") for s in ((3,), (3,), ())]
        snap = torch.empty(c.snapshot_bytes() // 8 + 1, dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        c.snapshot(snap)
        for k in range(repeats):
            other.force(every, *big)
            c.restore(snap)  # no noise estimates again
            c.predict(0.0)
            c.force(idx, *[x[k] for x in out])
        c.synchronize()
        other.synchronize()
        got = [x.cpu().numpy() for x in out]
    for x, y in zip(got, ref):
        x, y = x.reshape(repeats, rows, -1), y.reshape(1, rows, -1)
        err = np.linalg.norm(x - y, axis=2) / np.linalg.norm(y, axis=2)
        assert err.max() < 1e-6


@pytest.mark.parametrize("n,n_act", [(8192, 1), (8192, 33), (2000, 300), (1000, 37)])
def test_guarded_blocks_are_double_single(gpu, orc, n, n_act):
    """With the guard on for every listed particle each pair is double-single,
    also those of a far tile, which one warp takes whole: the DS result.  (Pair
    terms agree to ~2^-44, and the sums cancel to 1 % at worst: 1e-11.)"""
    eps = 4.0 / n
    m, r, v = ics.plummer(n, 40 + n)
    a, j, _ = orc.force(m, r, v, eps, nthreads=os.cpu_count() or 1)
    idx = ics.permutation(n, 8)[:n_act].astype(np.int32)
    res, unguarded = [], []
    for prec in ("hybrid", "ds"):
        with gpu.Context(prec) as c:
            c.set_state(m, r, v, a, j, np.zeros(n), np.full(n, 2.0 ** -30), eps, 0.02)
            c.predict(0.0)
            unguarded.append(c.force(idx))  # leaves the noise estimates
            res.append(c.force(idx))
    assert not np.array_equal(unguarded[0][0], res[0][0])
    for x, y in zip(*res):
        x, y = x.reshape(n_act, -1), y.reshape(n_act, -1)
        assert (np.linalg.norm(x - y, axis=1) / np.linalg.norm(y, axis=1)).max() < 1e-11
