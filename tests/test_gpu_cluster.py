"""Small lattices, several steps per launch as one cluster of blocks, against the oracle bit
for bit: one block and two, the cluster sizes' and block shapes' edges, the largest lattice a
cluster holds and one node more (the grid barrier); an overflow that one block marks for the
others in the middle of a launch."""
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


@pytest.mark.parametrize("lattice,Lx,Ly", [(1, L, 1) for L in (127, 128, 129, 1025, 2048, 2049, 4096, 4097)] +
                         [(q, *e) for q in (2, 3) for e in ((16, 8), (43, 3), (64, 32), (683, 3), (64, 64), (241, 17))])
def test_edges(B, lattice, Lx, Ly):
    cfg = dict(lattice=lattice, Lx=Lx, Ly=Ly, omega_eff=1.6, seed=5, replica=7)
    s0 = inputs.random_state(Q[lattice], Ly, Lx, 25.0, seed=Lx + Ly, hot=2, hot_value=300)
    with B.Lattice(**cfg) as lat:
        lat.set_step_kernel(2)
        lat.set_state(s0, 3)
        lat.step(2)
        lat.step(9)
        got, t = lat.get_state()
    assert t == 14 and np.array_equal(got, O.Lattice(**cfg).run(s0, 3, 11))


def heap(lattice, Lx, Ly):
    """Nodes nearly as full as a rest velocity may be, 99 % (D1Q3) or 98 % of a node's
    particles resting."""
    s0 = np.full((Q[lattice], Ly, Lx), 3, np.uint16)
    at = (slice(10, 22), slice(10, 22)) if lattice != 1 else (slice(0, 1), slice(260, 290))
    s0[(0,) + at] = (66000 if lattice == 1 else 66700) - 1000 * (Q[lattice] - 1)
    s0[(slice(1, None),) + at] = 1000
    return s0


@pytest.mark.parametrize("lattice,Lx,Ly,seed", [(1, 600, 1, 1), (2, 64, 60, 1)])
def test_overflow_marked_by_one_block(B, lattice, Lx, Ly, seed):
    cfg = dict(lattice=lattice, Lx=Lx, Ly=Ly, omega_eff=1.0, theta=0.01, seed=seed)
    s0 = heap(lattice, Lx, Ly)
    ref = O.Lattice(**cfg)
    cur, fail_t = s0, None
    for t in range(12):
        try:
            cur = ref.step(cur, t)
        except OverflowError:
            fail_t = t
            break
    assert fail_t is not None and fail_t >= 1
    with B.Lattice(**cfg) as lat:
        lat.set_step_kernel(2)
        lat.set_state(s0, 0)
        with pytest.raises(B.IlgError) as e:
            lat.step(12)
        assert e.value.status == B.ILG_E_OVERFLOW
        got, t = lat.get_state()
        assert t == fail_t and np.array_equal(got, cur)


@pytest.mark.parametrize("lattice,Lx,Ly", [(1, 255, 1), (1, 257, 1), (2, 64, 64), (2, 241, 17), (3, 43, 41), (3, 64, 64)])
def test_comparator_several_steps_at_once(B, lattice, Lx, Ly):
    """One call of 11 steps and eleven calls of one step (plain launches): the same doubles."""
    states = []
    f0 = np.random.default_rng(Lx).uniform(1.0, 30.0, (Q[lattice], Ly, Lx))
    for calls in ((11,), (1,) * 11):
        with B.LB(lattice, Lx, Ly, omega_j=1.7, omega=0.3) as lb:
            lb.set_state(f0)
            for T in calls:
                lb.step(T)
            states.append(lb.get_state()[0])
    assert np.array_equal(states[0], states[1])
