"""The force launches of a block step, counted in a captured graph.

HYBRID on a grid of one CTA per SM keeps its two builds apart; with more, up to 8192
particles, the small-block build serves every block in one launch.

An ensemble has one i-tile for blocks of every size.  A MIXED context's default
large variant has another (two i per lane), so nb_set_ensemble replaces it, and
with it everything that was chosen for it: the two variants are then one shape,
which is one launch, also for a single system loaded afterwards."""
import ctypes

import numpy as np
import pytest

from paper_1104_2700_gb300 import ics

pytestmark = pytest.mark.gpu


def _nodes(torch, stream, step):
    """Nodes of the graph that `step` leaves in `stream`."""
    cuda = ctypes.CDLL("libcuda.so.1")
    torch.cuda.synchronize()
    s, g, n = ctypes.c_void_p(stream.cuda_stream), ctypes.c_void_p(), ctypes.c_size_t()
    assert cuda.cuStreamBeginCapture_v2(s, 1) == 0  # thread local
    step()
    assert cuda.cuStreamEndCapture(s, ctypes.byref(g)) == 0
    assert cuda.cuGraphGetNodes(g, None, ctypes.byref(n)) == 0
    cuda.cuGraphDestroy(g)
    return n.value


def test_mixed_variants_become_one(gpu):
    torch = pytest.importorskip("torch")
    off, m, r, v, eps = ics.ensemble(5, 4, 7, 100, 300)[1:]
    m1, r1, v1 = ics.plummer(3000, 2)
    stream = torch.cuda.Stream()
    with gpu.Context("mixed", stream=stream) as c:
        c.set_particles(m1, r1, v1, 0.01, 0.02)
        # select, prediction, two force branches, corrector
        assert _nodes(torch, stream, lambda: c.block_step(1.0)) == 5
        c.set_ensemble(off, m, r, v, eps, 0.02)
        # next times, block list with the plan, prediction, force, corrector
        assert _nodes(torch, stream, lambda: c.block_step(1.0)) == 5
        c.set_particles(m1, r1, v1, 0.01, 0.02)
        assert _nodes(torch, stream, lambda: c.block_step(1.0)) == 4
        c.block_step(1.0)
        c.synchronize()


@pytest.mark.parametrize("ctas,nodes", [(0, 4), (2, 4), (1, 5)])
def test_hybrid_builds(gpu, ctas, nodes):
    torch = pytest.importorskip("torch")
    m, r, v = ics.plummer(3000, 2)
    stream = torch.cuda.Stream()
    with gpu.Context("hybrid", stream=stream, ctas_per_sm=ctas) as c:
        c.set_particles(m, r, v, 0.01, 0.02)
        # select, prediction, one force launch or two, corrector
        assert _nodes(torch, stream, lambda: c.block_step(1.0)) == nodes
        c.block_step(1.0)
        c.synchronize()
