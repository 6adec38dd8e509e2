"""The FP16 forms round alike one and two nodes per thread (launch.h, pair_pays):
the batch's persistent kernel, which steps pairs at every size, against the lone
lattice, which steps single nodes below 100,000 nodes (F16R: 48,000) and pairs
above, bit for bit over plain and check steps."""
import numpy as np
import pytest

from paper_1908_05396_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

P, WA, L = wl.PERIODIC, wl.WALL, wl.LID
_SINGLE = [(31, 30, 29), (8, 41, 9), (32, 17, 33)]
_PAIRS = [(61, 50, 47), (60, 53, 47)]
_FLOWS = {
    "lid": dict(face=(WA, WA, WA, L, WA, WA), U_lid=(0.05, 0.0, 0.02)),
    "forced": dict(face=(P, P, WA, WA, P, P), body_force=(1e-5, 2e-6, -3e-6)),
}


@pytest.fixture(scope="module")
def clbm():
    from paper_1908_05396_gb300 import build
    build.build()
    from paper_1908_05396_gb300 import clbm as c
    c.lib()
    return c


@pytest.mark.parametrize("n", [0.7, 1.0])
@pytest.mark.parametrize("flow", sorted(_FLOWS))
@pytest.mark.parametrize("dims", _SINGLE + _PAIRS)
@pytest.mark.parametrize("form", ["f16s", "f16s_sr", "f16r"])
def test_lone_lattice_and_pair_kernel_round_alike(clbm, form, dims, flow, n):
    dtype = form.partition("_")[0]
    lats = []
    for _ in range(2):
        lat = clbm.Lattice(*dims, K=0.02, n=n, dtype=dtype, check_interval=4, **_FLOWS[flow])
        if form == "f16s_sr":
            lat.set_rounding("stochastic")
        if not lats:
            f = lat.get_state() * (1 + wl.noise((19,) + lat.shape, seed=5, amp=0.02))
        lat.set_state(f)
        lats.append(lat)
    lats[0].step(9)
    with clbm.Batch(dtype, capacity=1, check_interval=4) as b:
        b.set_launch(32, 4, 1, 8)
        b.add(lats[1])
        b.step(9)
    assert np.array_equal(lats[0].get_state(), lats[1].get_state())
    for lat in lats:
        lat.close()
