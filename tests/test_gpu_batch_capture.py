"""Steps of an untuned batch of large lattices that a caller captures into a graph
of its own: every replay advances the lattices as fresh steps would, with new
random bits where stores are rounded stochastically.  And such a batch on the
legacy default stream, which cannot be captured: it never replays a graph."""
import numpy as np
import pytest

from paper_1908_05396_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def clbm():
    from paper_1908_05396_gb300 import build
    build.build()
    from paper_1908_05396_gb300 import clbm as c
    c.lib()
    return c


@pytest.mark.parametrize("form", ["f64", "f32", "f16s", "f16s_sr", "f16r"])
def test_replays_continue_the_steps(clbm, form):
    torch = pytest.importorskip("torch")
    dtype = form.partition("_")[0]

    def make(k):
        lat = clbm.Lattice(*((47, 46, 50), (60, 41, 43))[k], face=wl.CAVITY_FACES, K=0.02, n=0.7,
                           U_lid=(0.05, 0.0, 0.0), dtype=dtype)
        if form == "f16s_sr":
            lat.set_rounding("stochastic")
        return lat

    lone, mem = [make(0), make(1)], [make(0), make(1)]
    mem[1].step(5)                               # another step count than the batch's
    stream = torch.cuda.Stream()
    with clbm.Batch(dtype, capacity=2, stream=stream.cuda_stream) as b:
        for m in mem:
            b.add(m)
        b.step(2)
        b.sync()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=stream, capture_error_mode="thread_local"):
            b.step(4)
        with torch.cuda.stream(stream):
            for _ in range(3):
                g.replay()
        b.step(2)                                # and steps after them go on from there
        b.sync()
        for lat, n in zip(lone, (16, 21)):
            lat.step(n)
        for m, lat in zip(mem, lone):
            assert np.array_equal(m.get_state(), lat.get_state())
    for lat in lone + mem:
        lat.close()


@pytest.mark.parametrize("form", ["f32", "f16r"])
def test_legacy_default_stream(clbm, form):
    kw = dict(face=wl.CAVITY_FACES, K=0.02, n=0.7, U_lid=(0.05, 0.0, 0.0), dtype=form)
    with clbm.Lattice(47, 46, 50, **kw) as lat, clbm.Lattice(47, 46, 50, **kw) as lone:
        with clbm.Batch(form, capacity=1, stream=1) as b:      # cudaStreamLegacy
            b.add(lat)
            for _ in range(15):                  # past the steps launched singly
                b.step(10)
            b.sync()
        lone.step(150)
        assert np.array_equal(lat.get_state(), lone.get_state())
