"""Node-parallel steps, several per launch (candidate 2 on D1Q3 and D2Q5): the warp's
collision and the barrier between steps, against the oracle bit for bit at the sizes and
occupations where they can go wrong: lanes without a node, one and several blocks, rows
of odd length, occupations and removals on both sides of every chunk and group limit,
more extension words than a lane's ring holds, probabilities of 0 and 1, an overflow in
the middle of a launch."""
import numpy as np
import pytest

import oracle as O
from paper_2203_01380_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    from paper_2203_01380_gb300 import binding
    return binding


def check(B, cfg, s0, steps, t0=5):
    with B.Lattice(**cfg) as lat:
        lat.set_step_kernel(2)
        lat.set_state(s0, t0)
        lat.step(steps)
        got, t = lat.get_state()
    assert t == t0 + steps
    assert np.array_equal(got, O.Lattice(**cfg).run(s0, t0, steps))


@pytest.mark.parametrize("lattice,Lx,Ly", [(2, 3, 3), (2, 31, 3), (2, 32, 4), (2, 33, 5), (2, 43, 3), (2, 129, 7),
                                           (2, 152, 128), (2, 173, 113), (1, 3, 1), (1, 33, 1), (1, 128, 1),
                                           (1, 4097, 1), (1, 152 * 128 + 1, 1), (1, 152 * 512 + 33, 1)])
@pytest.mark.parametrize("omega,mean", [(1.7, 9.0), (0.5, 60.0)])
def test_extents(B, lattice, Lx, Ly, omega, mean):
    Q = 3 if lattice == 1 else 5
    s0 = inputs.random_state(Q, Ly, Lx, mean, seed=Lx * 7 + Ly)
    check(B, dict(lattice=lattice, Lx=Lx, Ly=Ly, omega_eff=omega, seed=11, replica=2), s0, 6)


@pytest.mark.parametrize("lattice", [1, 2])
@pytest.mark.parametrize("omega,theta", [(0.9, 1.0 / 3.0), (1.0, 0.4), (2.0, 1.0 / 3.0), (0.3, 0.5), (1.95, 0.1)])
@pytest.mark.parametrize("mean,hot", [(62.5, 0), (126.0, 0), (30.0, 5), (600.0, 2)])
def test_occupations(B, lattice, omega, theta, mean, hot):
    """Means around one and two chunks of 63; a few nodes with 13000 per velocity among
    ordinary ones (their lanes loop while the warp's others are done); 600 per velocity
    (several rings of extension words)."""
    Q = 3 if lattice == 1 else 5
    s0 = inputs.random_state(Q, 3, 37, mean, seed=int(mean), hot=hot, hot_value=13000)
    if lattice == 1:
        s0 = s0[:, :1]
    Ly = 1 if lattice == 1 else 3
    check(B, dict(lattice=lattice, Lx=37, Ly=Ly, omega_eff=omega, theta=theta, seed=13, replica=1), s0, 4)


@pytest.mark.parametrize("seed", [0, 2])
@pytest.mark.parametrize("kernel", [2, -1])
def test_overflow_in_the_middle_of_a_launch(B, kernel, seed):
    """A block of nodes holding nearly as much as their rest velocity may (98 % of a node's
    particles rest): one of them overflows after one or two steps of a twelve-step launch,
    as the oracle names it.  The context holds the state before that step and steps on
    from another state."""
    Lx, Ly = 40, 36
    cfg = dict(lattice=2, Lx=Lx, Ly=Ly, omega_eff=1.0, theta=0.01, seed=seed)
    s0 = np.full((5, Ly, Lx), 3, np.uint16)
    s0[0, 10:22, 10:22] = 66700 - 4000
    s0[1:, 10:22, 10:22] = 1000
    ref = O.Lattice(**cfg)
    cur, fail_t = s0, None
    for t in range(12):
        try:
            cur = ref.step(cur, t)
        except OverflowError:
            fail_t = t
            break
    assert fail_t is not None and fail_t >= 1
    small = inputs.random_state(5, Ly, Lx, 5.0, seed=9)
    with B.Lattice(**cfg) as lat:
        lat.set_step_kernel(kernel)
        lat.set_state(s0, 0)
        with pytest.raises(B.IlgError) as e:
            lat.step(12)
        assert e.value.status == B.ILG_E_OVERFLOW
        got, t = lat.get_state()
        assert t == fail_t and np.array_equal(got, cur)
        lat.set_state(small, 7)
        lat.step(3)
        got, t = lat.get_state()
    assert t == 10 and np.array_equal(got, ref.run(small, 7, 3))
