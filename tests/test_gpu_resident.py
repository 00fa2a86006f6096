"""Steps with the planes in the shared memory of all SMs, against the oracle bit for bit: shares
of one run, at the edges of the block shapes (4 and 16 runs of 32 nodes), rows shorter and longer
than a share, the narrowest rows it takes and narrower ones, launches of the fewest steps it takes
and fewer; an overflow that rolls back to the state before it although the shares have gone on;
and more steps than the mailbox has tags, against the same steps in launches too short for it."""
import numpy as np
import pytest

import oracle as O
from paper_2203_01380_gb300 import inputs

pytestmark = pytest.mark.gpu

Q = {1: 3, 2: 5, 3: 9}


@pytest.fixture(scope="module")
def B():
    from paper_2203_01380_gb300 import binding
    return binding


@pytest.mark.parametrize("lattice,Lx,Ly,omega", [
    (1, 8193, 1, 1.7), (1, 9999, 1, 0.6), (1, 19457, 1, 1.5), (1, 77826, 1, 1.2), (1, 160003, 1, 1.8),
    (2, 100, 100, 1.5), (2, 33, 251, 0.7), (2, 32, 257, 1.6), (2, 31, 300, 1.6), (2, 3001, 3, 1.6), (2, 139, 140, 1.4),
    (2, 301, 200, 1.9), (2, 279, 279, 0.5), (2, 401, 399, 1.5),
    (3, 32, 260, 1.5), (3, 95, 97, 0.7), (3, 1300, 9, 1.6), (3, 139, 141, 1.5), (3, 281, 277, 1.8), (3, 300, 290, 1.5),
])
def test_shares(B, lattice, Lx, Ly, omega):
    cfg = dict(lattice=lattice, Lx=Lx, Ly=Ly, omega_eff=omega, seed=3, replica=1)
    s0 = inputs.random_state(Q[lattice], Ly, Lx, 25.0, seed=Lx + 3 * Ly, hot=3, hot_value=500)
    ref = O.Lattice(**cfg)
    with B.Lattice(**cfg) as lat:
        lat.set_step_kernel(2)
        lat.set_state(s0, 7)
        t, want = 7, s0
        for n in (4, 9, 3):
            lat.step(n)
            want = ref.run(want, t, n)
            t += n
            got, gt = lat.get_state()
            assert gt == t and np.array_equal(got, want)


@pytest.mark.parametrize("lattice,Lx,Ly,before", [(1, 12000, 1, 0), (1, 12000, 1, 5), (2, 130, 66, 0), (2, 350, 60, 1)])
def test_overflow_rolls_back(B, lattice, Lx, Ly, before):
    # nodes nearly as full as a rest velocity may be; nearly all removed particles rest again
    cfg = dict(lattice=lattice, Lx=Lx, Ly=Ly, omega_eff=0.99, theta=0.01, seed=1)
    s0 = np.full((Q[lattice], Ly, Lx), 3, np.uint16)
    at = (slice(10, 22), slice(10, 22)) if lattice != 1 else (slice(0, 1), slice(260, 290))
    s0[(0,) + at] = (66000 if lattice == 1 else 66700) - 1000 * (Q[lattice] - 1)
    s0[(slice(1, None),) + at] = 1000
    ref = O.Lattice(**cfg)
    states, fail_t = [s0], None
    for t in range(14):
        try:
            states.append(ref.step(states[-1], t))
        except OverflowError:
            fail_t = t
            break
    assert fail_t is not None and fail_t >= 2
    with B.Lattice(**cfg) as lat:
        lat.set_step_kernel(2)
        lat.set_state(s0, 0)
        if before:
            lat.step(before)
        with pytest.raises(B.IlgError):
            lat.step(30)
        got, t = lat.get_state()
        assert t == fail_t and np.array_equal(got, states[fail_t])
        # and it goes on from there: the same step fails again, the state stays
        with pytest.raises(B.IlgError):
            lat.step(30)
        again, t = lat.get_state()
    assert t == fail_t and np.array_equal(again, got)


def test_more_steps_than_tags(B):
    cfg = dict(lattice=1, Lx=8200, Ly=1, n0=4.0, omega_eff=1.8, seed=8)
    steps = 66000
    with B.Lattice(**cfg) as a, B.Lattice(**cfg) as b:
        for lat in (a, b):
            lat.set_step_kernel(2)
            lat.init()
        a.step(steps - 500)
        a.step(500)
        for _ in range(steps // 3):
            b.step(3)
        sa, ta = a.get_state()
        sb, tb = b.get_state()
    assert ta == tb == steps and np.array_equal(sa, sb)
