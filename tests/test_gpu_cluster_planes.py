"""Small lattices whose planes stay in a cluster's shared memory for all steps of a launch,
against the oracle bit for bit: the edges of the block shapes beyond those of 256 threads, the
largest lattice a cluster holds and one node more, lattices whose last block is nearly empty,
one to a few steps (the state ends in either buffer), an overflow in the middle of a launch that
rolls back to the state before it, from either buffer, and a state that other calls read after."""
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


@pytest.mark.parametrize("omega", [0.6, 1.7])
@pytest.mark.parametrize("lattice,Lx,Ly", [(1, L, 1) for L in (3, 33, 1600, 4097, 7681, 8192, 8193)] +
                         [(q, *e) for q in (2, 3) for e in ((40, 40), (3, 3), (5, 821), (128, 64), (2731, 3))])
def test_edges(B, lattice, Lx, Ly, omega):
    cfg = dict(lattice=lattice, Lx=Lx, Ly=Ly, omega_eff=omega, seed=9, replica=2)
    s0 = inputs.random_state(Q[lattice], Ly, Lx, 30.0, seed=Lx * 7 + Ly, hot=3, hot_value=400)
    ref = O.Lattice(**cfg)
    with B.Lattice(**cfg) as lat:
        lat.set_step_kernel(2)
        lat.set_state(s0, 11)
        t, want = 11, s0
        for n in (2, 3, 1, 4):
            lat.step(n)
            want = ref.run(want, t, n)
            t += n
            got, gt = lat.get_state()
            assert gt == t and np.array_equal(got, want)
        assert lat.observables([(1, 0)])["mass"] == int(s0.sum())


@pytest.mark.parametrize("lattice,Lx,Ly,before", [(1, 600, 1, 0), (1, 600, 1, 1), (2, 64, 60, 0), (2, 120, 66, 1)])
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
            lat.step(20)
        got, t = lat.get_state()
    assert t == fail_t and np.array_equal(got, states[fail_t])
