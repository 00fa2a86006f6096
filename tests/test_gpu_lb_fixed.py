"""The comparator's fixed-point relaxation at the edges of its domain, one step against the
update written per velocity in extended precision: weights and rates at the ends of their ranges
(1 - omega and 1 - omega^j of both signs, 0 and 1), results that fall below the least size it
takes, turn negative or pass the largest, and values that differ by the most bits it takes and
by one more.  The domain's inside is also held to one rounding of the result."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

LD = np.longdouble
VEL = {1: [(0, 0), (1, 0), (-1, 0)],
       2: [(0, 0), (1, 0), (-1, 0), (0, 1), (0, -1)],
       3: [(0, 0), (1, 0), (-1, 0), (0, 1), (0, -1), (1, 1), (-1, -1), (1, -1), (-1, 1)]}
THETA = {1: [1e-6, 1 / 3, 1 - 1e-6], 2: [1e-6, 1 / 3, 0.5], 3: [1e-6, 1 / 3, 1 - 1e-6]}


@pytest.fixture(scope="module")
def B():
    from paper_2203_01380_gb300 import binding
    return binding


def one_step(lattice, f, oj, om, theta):
    t, v = LD(theta), VEL[lattice]
    w = {1: [1 - t] + [t / 2] * 2, 2: [1 - 2 * t] + [t / 2] * 4,
         3: [(1 - t) ** 2] + [t * (1 - t) / 2] * 4 + [t * t / 4] * 4}[lattice]
    f = f.astype(LD)
    rho = f.sum(0)
    out, size = np.empty_like(f), np.empty_like(f)
    for i in range(len(v)):
        j = 0 if i == 0 else (i + 1 if i % 2 else i - 1)
        even, odd = (1 - LD(om)) * (f[i] + f[j]) / 2, (1 - LD(oj)) * (f[i] - f[j]) / 2
        p, s = LD(om) * w[i] * rho + even + odd, LD(om) * w[i] * rho + f[i] + f[j]
        out[i], size[i] = (np.roll(a, (v[i][1], v[i][0]), (0, 1)) for a in (p, s))
    return out, size


@pytest.mark.parametrize("oj,om", [(1.9, 0.1), (0.3, 1.99), (2.0, 2.0), (0.0, 0.0), (1.0, 1.0), (1.0, 0.5),
                                   (1.0 + 2**-52, 1.0 - 2**-53), (2.0, 1e-15)])
@pytest.mark.parametrize("lattice", [1, 2, 3])
def test_edges_of_the_domain(B, lattice, oj, om):
    Q = len(VEL[lattice])
    rng = np.random.default_rng(100 * lattice + int(10 * oj))
    Lx, Ly = (900, 1) if lattice == 1 else (37, 29)
    for theta in THETA[lattice]:
        # one velocity up to 2^11 times smaller or larger than the others, others alike
        f = rng.uniform(1.0, 2.0, (Q, Ly, Lx))
        pick = rng.integers(0, Q, (Ly, Lx))
        scale = 2.0 ** rng.integers(-11, 12, (Ly, Lx))
        f[pick, np.arange(Ly)[:, None], np.arange(Lx)] *= scale
        with B.LB(lattice, Lx, Ly, n0=1.0, omega_j=oj, omega=om, theta=theta) as lb:
            lb.set_state(f)
            lb.step(1)
            got, _ = lb.get_state()
        want, size = one_step(lattice, f, oj, om, theta)
        # outside: the weights (2 roundings), the density (Q - 1), two products, two sums, of
        # at most the terms' sum each
        err = np.abs(got.astype(LD) - want)
        assert np.all(err <= (Q + 6) * 2.0**-53 * size)


@pytest.mark.parametrize("oj,om", [(1.8, 0.2), (0.7, 0.7), (1.3, 0.7)])
@pytest.mark.parametrize("lattice", [1, 2, 3])
def test_one_rounding_inside(B, lattice, oj, om):
    Q = len(VEL[lattice])
    rng = np.random.default_rng(lattice)
    Lx, Ly = (900, 1) if lattice == 1 else (37, 29)
    theta = 0.25  # the weights are exact doubles
    f = rng.uniform(1.0, 2.0, (Q, Ly, Lx))
    with B.LB(lattice, Lx, Ly, n0=1.0, omega_j=oj, omega=om, theta=theta) as lb:
        lb.set_state(f)
        lb.step(1)
        got, _ = lb.get_state()
    want, _ = one_step(lattice, f, oj, om, theta)
    # half a unit of the result's last bit, and four products that lack up to two units of 2^-60
    # (D2Q9: 2^-58) of the largest value each
    units = 8 * 2.0 ** (-58 if Q == 9 else -60) * 2.0
    assert np.all(np.abs(got.astype(LD) - want) <= 2.0**-53 * 2.0 ** np.ceil(np.log2(want.astype(float))) + units)


@pytest.mark.parametrize("lattice,Lx,Ly", [(1, 63, 1), (1, 1025, 1), (1, 4097, 1), (1, 16384, 1), (1, 16385, 1),
                                           (2, 3, 3), (2, 65, 63), (2, 91, 90), (2, 128, 128), (2, 129, 128),
                                           (3, 7, 9), (3, 128, 64), (3, 91, 91)])
def test_steps_in_a_cluster(B, lattice, Lx, Ly):
    """Many steps in one launch (lattices that a cluster's shared memory holds, and one node or row
    more) against the same steps one call at a time, bit for bit, ending in either buffer."""
    kw = dict(n0=30.0, amp=20.0, mode_mx=1, omega_j=1.7, omega=0.3)
    with B.LB(lattice, Lx, Ly, **kw) as a, B.LB(lattice, Lx, Ly, **kw) as b:
        a.init()
        b.init()
        for n in (2, 5):
            a.step(n)
            for _ in range(n):
                b.step(1)
            fa, ta = a.get_state()
            fb, tb = b.get_state()
            assert ta == tb and np.array_equal(fa, fb)
        assert a.observables([(1, 0)])["mass"] == b.observables([(1, 0)])["mass"]
