"""The comparator's step where its integer density sums begin and end: nodes whose velocities
are alike (summed in integers), that differ by every power of two around the limit, that hold
zeros, negative, subnormal and very large values (summed in fp64), rates whose weights leave
the integer path (omega = 0); one step against the update written per velocity in numpy, with
the error of a handful of roundings of its terms; and many steps in one call against the same
steps one call at a time, bit for bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

VEL = {1: [(0, 0), (1, 0), (-1, 0)],
       2: [(0, 0), (1, 0), (-1, 0), (0, 1), (0, -1)],
       3: [(0, 0), (1, 0), (-1, 0), (0, 1), (0, -1), (1, 1), (-1, -1), (1, -1), (-1, 1)]}
WEIGHTS = {1: [2 / 3, 1 / 6, 1 / 6], 2: [1 / 3] + [1 / 6] * 4, 3: [4 / 9] + [1 / 9] * 4 + [1 / 36] * 4}


@pytest.fixture(scope="module")
def B():
    from paper_2203_01380_gb300 import binding
    return binding


def one_step(lattice, f, oj, om):
    """The update and, per value, the sum of its terms' magnitudes."""
    w, v = WEIGHTS[lattice], VEL[lattice]
    rho, mag = f.sum(0), np.abs(f).sum(0)
    out, size = np.empty_like(f), np.empty_like(f)
    for i in range(len(w)):
        j = 0 if i == 0 else (i + 1 if i % 2 else i - 1)
        p = om * w[i] * rho + (1 - om) * 0.5 * (f[i] + f[j]) + (1 - oj) * 0.5 * (f[i] - f[j])
        s = om * w[i] * mag + np.abs(f[i]) + np.abs(f[j])
        out[i], size[i] = (np.roll(a, (v[i][1], v[i][0]), (0, 1)) for a in (p, s))
    return out, size


def states(lattice, Ly, Lx):
    rng = np.random.default_rng(lattice)
    Q = len(WEIGHTS[lattice])
    alike = rng.uniform(1.0, 2.0, (Q, Ly, Lx))
    spread = alike * 2.0 ** rng.integers(-13, 1, (Q, Ly, Lx))
    odd = rng.choice([0.0, 1.0, -3.0, 1e-310, 1e-30, 7e5, 1e150, 0.1], (Q, Ly, Lx)) * alike
    ties = np.round(alike * 2 ** 52) / 2 ** 52 + 2.0 ** rng.integers(0, 4, (Q, Ly, Lx))
    return dict(alike=alike, spread=spread, odd=odd, ties=ties, tiny=alike * 1e-200, huge=alike * 1e200)


@pytest.mark.parametrize("name", ["alike", "spread", "odd", "ties", "tiny", "huge"])
@pytest.mark.parametrize("oj,om", [(1.8, 0.2), (0.7, 0.7), (2.0, 0.0), (1.0, 1.0)])
@pytest.mark.parametrize("lattice,Lx,Ly", [(1, 1030, 1), (2, 61, 43), (3, 40, 33)])
def test_one_step(B, lattice, Lx, Ly, oj, om, name):
    f = states(lattice, Ly, Lx)[name]
    with B.LB(lattice, Lx, Ly, n0=1.0, omega_j=oj, omega=om) as lb:
        lb.set_state(f, 3)
        lb.step(1)
        got, t = lb.get_state()
    want, size = one_step(lattice, f, oj, om)
    assert t == 4
    # about six roundings on each side, each half a unit of 2^-52 of at most the terms' sum
    assert np.all(np.abs(got - want) <= 12 * 2.0 ** -53 * size + 1e-320)


@pytest.mark.parametrize("lattice,Lx,Ly", [(1, 700, 1), (2, 130, 70), (3, 65, 64), (2, 1600, 1400)])
def test_steps_in_one_launch(B, lattice, Lx, Ly):
    kw = dict(n0=30.0, amp=20.0, mode_mx=1, omega_j=1.7, omega=0.3)
    with B.LB(lattice, Lx, Ly, **kw) as a, B.LB(lattice, Lx, Ly, **kw) as b:
        a.init()
        b.init()
        a.step(7)
        for _ in range(7):
            b.step(1)
        fa, ta = a.get_state()
        fb, tb = b.get_state()
    assert ta == tb == 7 and np.array_equal(fa, fb)
