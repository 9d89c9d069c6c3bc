"""nb_force into a caller's device arrays: every combination of wanted outputs
and an array at an odd byte offset (which takes a copy) give the bits of the
call that asks for all of them."""
import ctypes

import numpy as np
import pytest

from paper_1104_2700_gb300 import ics

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["hybrid", "mixed", "ds", "fp64"])
@pytest.mark.parametrize("n_act", [1, 33, 1500])
def test_outputs_wanted(gpu, prec, n_act):
    torch = pytest.importorskip("torch")
    n = 2000
    m, r, v = ics.plummer(n, 3)
    idx = torch.from_numpy(np.sort(ics.permutation(n, 8)[:n_act]).astype(np.int32)).cuda()
    p = lambda t: ctypes.c_void_p(t.data_ptr()) if t is not None else None  # noqa: E731
    with gpu.Context(prec) as c:
        c.set_particles(m, r, v, 4.0 / n, 0.02)
        snap = torch.empty(c.snapshot_bytes() // 8 + 1, dtype=torch.float64, device="cuda")
        c.snapshot(snap)  # (HYBRID keeps a noise estimate of each evaluation)

        def run(out):
            c.restore(snap)
            c.predict(0.0)
            assert gpu.nb_force(c.handle, n_act, p(idx), *[p(t) for t in out], 1) == 0
            c.synchronize()
            return out

        def fresh():
            return [torch.full((k * n_act,), 7.0, dtype=torch.float64, device="cuda")
                    for k in (3, 3, 1)]
        ref = run(fresh())
        for want in range(8):
            got = run([t if want >> k & 1 else None for k, t in enumerate(fresh())])
            for k in range(3):
                if want >> k & 1:
                    assert torch.equal(got[k], ref[k])
        raw = torch.zeros(8 * 3 * n_act + 16, dtype=torch.uint8, device="cuda")
        c.restore(snap)
        c.predict(0.0)
        assert gpu.nb_force(c.handle, n_act, p(idx), ctypes.c_void_p(raw.data_ptr() + 4), None,
                            None, 1) == 0
        c.synchronize()
        odd = raw[4:4 + 24 * n_act].cpu().numpy().tobytes()
        assert odd == ref[0].cpu().numpy().tobytes()
