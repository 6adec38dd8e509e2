"""The collision for unit rates omega_9..18 (the default) against the one for
any rates, which a lattice takes when a single rate differs from 1 in its last
bit: the two evaluate the same update, so they agree to rounding, in the
storage forms whose stored value is the deviation, with and without a body force, alone and in a batch that holds
lattices of both kinds.

Tolerances.  FP64: a population is below 0.5 and an update has under 500
roundings of 2^-53 at that scale, most of them far smaller: 1e-13 over 20
steps.  FP32: 2^-24 at the scale of a deviation (0.05), under 20 of them per
population and step: 1e-6 over 20 steps.  F16S: after one step the
two FP32 results straddle at most one rounding boundary of the stored value:
one FP16 ulp of the deviation (2^-10 of it, and 1e-7 near zero)."""
import numpy as np
import pytest

from paper_1908_05396_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

W = np.array([1 / 3] + [1 / 18] * 6 + [1 / 36] * 12)
_ONE = float(np.nextafter(1.0, 2.0))
_PROBS = {
    "cavity": wl.cavity(21, 100.0, 0.7, dims=(37, 21, 10)),
    "forced": wl.Problem("mixed", 33, 17, 9, (wl.WALL, wl.WALL, wl.WALL, wl.LID, wl.PERIODIC, wl.PERIODIC),
                         K=0.01, n=1.3, U_lid=(0.04, 0.0, 0.02), body_force=(1e-5, 2e-6, -2e-6)),
    "box": wl.Problem("box", 6, 5, 4, (wl.PERIODIC,) * 6, K=0.05, n=1.0, body_force=(1e-5, -2e-6, 3e-6)),
}


@pytest.fixture(scope="module")
def clbm():
    from paper_1908_05396_gb300 import build
    build.build()
    from paper_1908_05396_gb300 import clbm as c
    c.lib()
    return c


def _pair(clbm, prob, form, **kw):
    """Two lattices in the same state, the second with rates of 1 but for one last bit."""
    out = []
    for k in range(2):
        lat = clbm.Lattice(**prob.kwargs(), dtype=form, check_interval=10, **kw)
        f = lat.get_state() * (1 + wl.noise((19,) + lat.shape, seed=3, amp=0.02))
        lat.set_state(f)
        if k:
            lat.set_rates({12: _ONE})
        out.append(lat)
    return out


def _close(f, g, form):
    if form in ("f64", "f32"):
        assert np.abs(f - g).max() <= {"f64": 1e-13, "f32": 1e-6}[form]
    else:
        dev = np.abs(g - W[:, None, None, None])
        assert np.all(np.abs(f - g) <= dev * 2.0 ** -10 + 1e-7)


@pytest.mark.parametrize("name", sorted(_PROBS))
@pytest.mark.parametrize("form", ["f64", "f32", "f16s", "f32_inplace", "f64_inplace"])
def test_unit_rates_match_any_rates(clbm, form, name):
    form, _, inplace = form.partition("_")
    a, b = _pair(clbm, _PROBS[name], form, in_place=bool(inplace))
    n = 20 if form in ("f64", "f32") else 1
    for lat in (a, b):
        lat.step(n)
    _close(a.get_state(), b.get_state(), form)
    if form == "f64":
        for x, y in zip(a.fields(), b.fields()):
            assert np.abs(x - y).max() <= 1e-11
    a.close()
    b.close()


@pytest.mark.parametrize("form", ["f64", "f32", "f16s"])
def test_batch_of_both_kinds(clbm, form):
    # odd step counts and a full check interval; membership changes while it runs
    alone = {}
    for name, prob in _PROBS.items():
        for k, lat in enumerate(_pair(clbm, prob, form)):
            lat.step(1)
            alone[name, k] = lat.get_state()
            lat.close()
    lats = {(name, k): lat for name, prob in _PROBS.items()
            for k, lat in enumerate(_pair(clbm, prob, form))}
    with clbm.Batch(form, capacity=8, check_interval=10) as batch:
        slots = {key: batch.add(lat) for key, lat in lats.items()}
        batch.step(1)
        for key, lat in lats.items():
            _close(lat.get_state(), alone[key], form)
        for name in _PROBS:
            batch.remove(slots[name, 1])
        batch.step(19)
        for name in _PROBS:
            batch.add(lats[name, 1])
        batch.step(10)
        assert not batch.stats_all()["diverged"].any()
    for (name, k), lat in lats.items():
        assert lat.steps_done() == (30 if k == 0 else 11)
        lat.close()
