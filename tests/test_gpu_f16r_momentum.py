"""F16R stores remainders after a reference that the writer takes off the
moments and the reader puts back population by population: the two must cancel,
or every step drags the flow.  A uniform flow in a periodic box feels no shear,
so its mean momentum must stay.

Tolerance.  The remainders of u = 0.05 are below 0.5 (in units of 1/1024), so a
stochastically rounded store has a standard deviation of at most half of
2^-12, and ten populations carry x momentum: 3.8e-4 a node and step, against a
momentum of 51.  Over 2000 steps the mean over 32^3 nodes strays by
3.8e-4 sqrt(2000 / 32768) / 51 = 1.8e-6 in relation; five of that are 9e-6, and
1.5e-5 leaves room for FP32 roundings.  Constants that differ in their last bits,
3e-8 of the momentum a step, would make 4e-5 and more."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def clbm():
    from paper_1908_05396_gb300 import build
    build.build()
    from paper_1908_05396_gb300 import clbm as c
    c.lib()
    return c


# one node per thread, a pair per thread, pairs with a second node in the padding
@pytest.mark.parametrize("dims", [(32, 32, 32), (40, 40, 40), (41, 40, 39)])
@pytest.mark.parametrize("batched", [False, True])
def test_uniform_flow_keeps_its_momentum(clbm, dims, batched):
    import oracle
    ex = oracle.velocities()[:, 0]
    u = 0.05
    f = oracle.weights() * (1 + 3 * ex * u + 4.5 * (ex * u) ** 2 - 1.5 * u * u)
    with clbm.Lattice(*dims, face=(clbm.PERIODIC,) * 6, K=0.02, n=1.0, dtype="f16r") as lat:
        lat.set_state(np.broadcast_to(f[:, None, None, None], (19,) + lat.shape).copy())
        u0 = lat.fields()[1][0].mean()
        if batched:
            with clbm.Batch("f16r", capacity=1) as b:
                b.set_launch(32, 4, 1, 8)       # the batch's own kernel
                b.add(lat)
                b.step(2000)
        else:
            lat.step(2000)
        u1 = lat.fields()[1][0].mean()
    assert abs(u1 / u0 - 1) <= 1.5e-5
