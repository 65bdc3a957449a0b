"""Steps captured by the caller on the context's stream and replayed without
the library's knowledge: every reading call has to see the state of the last
replay, as if the steps had been called."""
import numpy as np
import pytest

from paper_2405_07898_gb300 import binding, inputs as I

pytestmark = pytest.mark.gpu


def capture(obj, nsteps):
    import torch

    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=obj.stream, capture_error_mode="thread_local"):
        obj.step(nsteps, 2.0)
    return g


def replay(g, stream):
    import torch

    with torch.cuda.stream(stream):
        g.replay()


@pytest.mark.parametrize("kw", [dict(persistent="on"), dict(persistent="off", use_graphs=False)])
def test_context(kw):
    s = I.bcc_cube(8, 600.0)
    with binding.MD(s, lanes_per_atom=2, **kw) as md, binding.MD(s, lanes_per_atom=2, **kw) as ref:
        g = capture(md, 7)
        for _ in range(4):
            replay(g, md.stream)
            ref.step(7, 2.0)
            assert md.energy() == ref.energy()
            np.testing.assert_array_equal(md.virial(), ref.virial())
            a, b = md.get_state(), ref.get_state()
            assert a[2] == b[2]
            for x, y in zip(a[:2], b[:2]):
                np.testing.assert_array_equal(x, y)
            assert md.stats()["rebuilds"] == ref.stats()["rebuilds"]
        del g


def test_batch():
    systems = [I.bcc_cube(6, 600.0), I.bcc_cube(8, 300.0)]
    with binding.MDBatch(systems, use_graphs=False) as b, binding.MDBatch(systems, use_graphs=False) as ref:
        g = capture(b, 7)
        for _ in range(4):
            replay(g, b.stream)
            ref.step(7, 2.0)
            for x, y in zip(b.energy(), ref.energy()):
                np.testing.assert_array_equal(x, y)
            for x, y in zip(b.get_state(1), ref.get_state(1)):
                np.testing.assert_array_equal(x, y)
            assert b.info()["steps"] == ref.info()["steps"]
        del g
