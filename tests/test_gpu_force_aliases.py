"""nb_force on device arrays that share memory, or end before the results do.

The results are as if they were copied out after the evaluation, acc, then jerk,
then pot: an array that shares bytes with the list or with an earlier array holds
the whole of what was written last, bit for bit, and an array that its allocation
cannot hold is refused."""
import ctypes

import numpy as np
import pytest

from paper_1104_2700_gb300 import ics

pytestmark = pytest.mark.gpu
N, K = 2000, 700


def _at(t, byte=0):
    return ctypes.c_void_p(t.data_ptr() + byte)


@pytest.fixture
def loaded(gpu):
    torch = pytest.importorskip("torch")
    m, r, v = ics.plummer(N, 3)
    idx = np.sort(ics.permutation(N, 8)[:K]).astype(np.int32)
    with gpu.Context("ds") as c:
        c.set_particles(m, r, v, 4.0 / N, 0.02)
        c.predict(0.0)
        out = [torch.empty(n * K, dtype=torch.float64, device="cuda") for n in (3, 3, 1)]
        lst = torch.from_numpy(idx).cuda()
        torch.cuda.synchronize()
        assert gpu.nb_force(c.handle, K, _at(lst), *[_at(t) for t in out], 1) == 0
        c.synchronize()
        yield torch, c, lst, out


@pytest.mark.parametrize("which", [0, 1, 2])
def test_result_over_the_list(gpu, loaded, which):
    torch, c, lst, ref = loaded
    buf = torch.zeros_like(ref[which])
    buf.view(torch.int32)[:K] = lst
    torch.cuda.synchronize()
    out = [_at(buf) if q == which else None for q in range(3)]
    assert gpu.nb_force(c.handle, K, _at(buf), *out, 1) == 0
    c.synchronize()
    assert torch.equal(buf, ref[which])


def test_results_over_each_other(gpu, loaded):
    torch, c, lst, ref = loaded
    buf = torch.zeros(4 * K, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    # acc at 0, jerk at K doubles, pot at the last K of jerk
    assert gpu.nb_force(c.handle, K, _at(lst), _at(buf), _at(buf, 8 * K), _at(buf, 24 * K), 1) == 0
    c.synchronize()
    want = torch.cat([ref[0][:K], ref[1][:2 * K], ref[2]])
    assert torch.equal(buf, want)


def test_array_too_short(gpu, loaded):
    """The last 24 bytes of an allocation, asked to take two rows."""
    torch, c, lst, ref = loaded
    cuda = ctypes.CDLL("libcuda.so.1")
    p = ctypes.c_uint64()
    assert cuda.cuMemAlloc_v2(ctypes.byref(p), ctypes.c_size_t(4096)) == 0
    end = p.value + 4096
    try:
        assert gpu.nb_force(c.handle, 1, _at(lst), ctypes.c_void_p(end - 24), None, None, 1) == 0
        c.synchronize()
        assert gpu.nb_force(c.handle, 2, _at(lst), ctypes.c_void_p(end - 24), None, None, 1) != 0
    finally:
        torch.cuda.synchronize()
        cuda.cuMemFree_v2(p)


def test_captured_call(gpu):
    """The call goes into a graph, captured in the strictest mode, and its
    replay writes the arrays again."""
    torch = pytest.importorskip("torch")
    m, r, v = ics.plummer(N, 3)
    s = torch.cuda.Stream()
    with gpu.Context("ds", stream=s) as c:
        c.set_particles(m, r, v, 4.0 / N, 0.02)
        lst = torch.arange(K, dtype=torch.int32, device="cuda")
        out = [torch.empty(n * K, dtype=torch.float64, device="cuda") for n in (3, 3, 1)]
        torch.cuda.synchronize()

        def call():
            c.predict(0.0)
            assert gpu.nb_force(c.handle, K, _at(lst), *[_at(t) for t in out], 1) == 0
        call()
        c.synchronize()
        want = [t.clone() for t in out]
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            call()
        for t in out:
            t.zero_()
        torch.cuda.synchronize()
        g.replay()
        torch.cuda.synchronize()
    for x, y in zip(out, want):
        assert torch.equal(x, y)
