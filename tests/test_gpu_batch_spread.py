"""A batch whose launch was neither set nor tuned steps large lattices by one
launch each, in replayed graphs: every lattice must advance exactly as it does
alone, over graph steps and single ones, check steps, members that join with
another step count and leave, check intervals of whole and short graphs, and a member that brings
the mean size below the rule's line and the batch back to its own kernel."""
import numpy as np
import pytest

from paper_1908_05396_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

P, WA, L = wl.PERIODIC, wl.WALL, wl.LID
SIZES = {"large": [(47, 46, 50), (53, 61, 37), (96, 33, 40)],
         "falls": [(47, 46, 50), (53, 61, 37), (72, 31, 22)]}


@pytest.fixture(scope="module")
def clbm():
    from paper_1908_05396_gb300 import build
    build.build()
    from paper_1908_05396_gb300 import clbm as c
    c.lib()
    return c


@pytest.mark.parametrize("sizes", sorted(SIZES))
@pytest.mark.parametrize("interval", [20, 14])
@pytest.mark.parametrize("form", ["f64", "f32", "f16s", "f16s_sr", "f16r"])
def test_untuned_batch_equals_lone(clbm, form, interval, sizes):
    def make(k):
        lat = clbm.Lattice(*SIZES[sizes][k], face=((WA, WA, WA, L, WA, WA), (P, P, P, P, WA, L),
                                                   (WA, WA, P, P, P, P))[k],
                           K=0.05, n=(0.8, 1.0, 1.2)[k], U_lid=None if k == 2 else (0.05, 0, 0),
                           body_force=(1e-5, 2e-6, 0.0) if k else None, dtype=form[:4].rstrip("_"),
                           check_interval=interval)
        if form == "f16s_sr":
            lat.set_rounding("stochastic")
        return lat

    lone, mem = [make(k) for k in range(3)], [make(k) for k in range(3)]
    mem[2].step(3)
    lone[2].step(3)
    with clbm.Batch(form[:4].rstrip("_"), capacity=3, check_interval=interval) as b:
        s0, s1 = b.add(mem[0]), b.add(mem[1])
        b.step(23)
        b.add(mem[2])
        b.step(145)
        b.remove(s1)
        b.step(161)
        st = b.stats(s0)
        assert st["steps"] == 329 and not st["diverged"]
        assert np.isfinite(st["residual"]) and abs(st["mass"] / lone[0].N - 1.0) < 1e-2
    for l, m, n in zip(lone, mem, (329, 168, 306)):
        l.step(n)
        for a, c in zip(l.fields(), m.fields()):
            assert np.array_equal(a, c)
        l.close()
        m.close()
