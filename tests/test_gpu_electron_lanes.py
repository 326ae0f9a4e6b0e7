"""The two launch forms of the electron integrators (four lanes an electron for few
electrons, one lane for many) and the two phase reductions (phases below and above
1e6), against the FP64 oracle and each other, for every wave."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu
EPS = oracle.eps_rr(0.8)


@pytest.fixture(scope="module")
def picrr():
    import __graft_entry__

    __graft_entry__.build()
    import paper_1008_1685_gb300 as m

    return m


def cases(n, x0=0.0):
    r = np.random.default_rng(n)
    return [dict(wave=i % 3, a0=float(r.uniform(5, 300)), tau=40.0, x0=x0, p0=tuple(float(v) for v in r.uniform(-50, 5, 3)))
            for i in range(n)]


def reference(c, integrator, rr, deriv, dt, n, every):
    kw = dict(every=every, eps=EPS, rr=rr, tau=c["tau"])
    if integrator == 0:
        return oracle.pw_leapfrog(c["wave"], c["a0"], c["x0"], np.array(c["p0"]), dt, n, **kw)
    return oracle.pw_rk4(c["wave"], c["a0"], c["x0"], np.array(c["p0"]), dt, n, deriv=deriv, **kw)


def off(a, b):
    return np.max(np.abs(a - b) / (np.max(np.abs(b), axis=0) + 1.0))


@pytest.mark.parametrize("integrator,rr,deriv", [(0, True, False), (0, False, False), (1, True, True), (1, True, False),
                                                 (1, False, False)])
def test_few_and_many_electrons_agree(picrr, integrator, rr, deriv):
    few = cases(37)  # four lanes an electron, a ragged warp of each kind
    many = few + cases(4900)  # one lane
    kw = dict(integrator=integrator, rr=rr, deriv=deriv, dt=0.01, nsteps=305, every=100)
    a, b = picrr.electron_scan(few, **kw), picrr.electron_scan(many, **kw)
    assert a.shape == (37, 3, 5) and b.shape == (4937, 3, 5)
    assert off(a, b[:37]) <= 1e-12
    for i in (0, 1, 2, 35, 36):
        assert off(a[i], reference(few[i], integrator, rr, deriv, 0.01, 305, 100)[:3]) <= 1e-9
    for i in (3000, 4935, 4936):
        assert off(b[i], reference(many[i], integrator, rr, deriv, 0.01, 305, 100)[:3]) <= 1e-9


@pytest.mark.parametrize("x0", [-2.0e6, -999_999.5])  # beyond the short reduction, and crossing into it
def test_large_phases(picrr, x0):
    """x is rounded to 2^-53 |x| = 1.2e-10 a step at these positions, on both sides: 200
    steps of it move the phase by at most 2.4e-8, momenta by that times a0 relative."""
    few = cases(6, x0)
    for integrator, deriv in ((0, False), (1, True)):
        a = picrr.electron_scan(few, integrator=integrator, rr=True, deriv=deriv, dt=0.01, nsteps=200, every=50)
        for i, c in enumerate(few):
            b = reference(c, integrator, True, deriv, 0.01, 200, 50)
            assert off(a[i][:, 2:], b[:, 2:]) <= 1e-5, (x0, integrator, i)


@pytest.mark.parametrize("pad", [0, 4900])  # four lanes an electron, one lane
@pytest.mark.parametrize("integrator,rr,deriv", [(0, True, False), (0, False, False), (1, True, True), (1, False, False)])
def test_no_field_outside_the_pulse_at_any_phase(picrr, integrator, rr, deriv, pad):
    """An electron that no pulse reaches keeps its momentum bit for bit: at infinite or undefined phases,
    and in a pulse so short that pi / tau is not finite."""
    far = [dict(wave=2, a0=100.0, tau=40.0, x0=x0, p0=(0.5, -0.25, 2.0)) for x0 in (np.inf, -np.inf, np.nan, 5.0)]
    short = dict(wave=2, a0=100.0, tau=1e-310, x0=0.0, p0=(0.0, 0.0, 0.0))
    out = picrr.electron_scan(far + [short] + cases(pad), integrator=integrator, rr=rr, deriv=deriv, dt=0.01, nsteps=9, every=3)
    assert np.all(out[:4, :, 2:] == (0.5, -0.25, 2.0)) and np.all(out[4, :, 1:] == 0.0)
    assert np.all(out[0, :, 1] == np.inf) and np.all(out[1, :, 1] == -np.inf) and np.all(np.isnan(out[2, :, 1]))


@pytest.mark.parametrize("pad", [0, 4900])
@pytest.mark.parametrize("a0", [1e3, 1e153, 1e155, 1e200])
def test_leapfrog_amplitudes_whose_square_overflows(picrr, a0, pad):
    """Without radiation reaction no product in the step needs the square of the field: 20 steps agree with the
    oracle's to a few roundings of 2^-53 a step, relative to the momenta's size."""
    few = [dict(wave=w, a0=a0, tau=0.19, x0=0.0, p0=(0.0, 0.0, 0.0)) for w in (0, 1, 2)]
    out = picrr.electron_scan(few + cases(pad), integrator=0, rr=False, dt=0.01, nsteps=20, every=1)
    for i, c in enumerate(few):
        b = reference(c, 0, False, False, 0.01, 20, 1)
        assert np.all(np.isfinite(b)) and np.max(np.abs(b[:, 2:])) > 1e-3 * a0
        assert off(out[i], b[:20]) <= 1e-13, (i, a0)
