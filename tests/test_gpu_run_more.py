"""Several steps per launch through the D2Q9 node-parallel kernel and the staged warp kernels,
against the oracle bit for bit: extents around a warp and a block, rows of whole and of ragged
tiles and of one vector, more tiles than warps, vectors with one node, some and all beyond the
fast collision, occupations on both sides of its limits, probabilities of 0 and 1, both
samplers; the default choice on either side of its limits."""
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


def check(B, cfg, s0, steps, kernel, t0=5):
    with B.Lattice(**cfg) as lat:
        lat.set_step_kernel(kernel)
        lat.set_state(s0, t0)
        lat.step(steps)
        got, t = lat.get_state()
    assert t == t0 + steps and np.array_equal(got, O.Lattice(**cfg).run(s0, t0, steps))


@pytest.mark.parametrize("Lx,Ly", [(3, 3), (31, 4), (33, 5), (128, 3), (152, 129), (311, 67)])
@pytest.mark.parametrize("omega,mean,sampler", [(1.7, 9.0, 0), (0.5, 60.0, 0), (1.0, 20.0, 0), (2.0, 70.0, 0), (1.4, 15.0, 1)])
def test_d2q9_node_parallel(B, Lx, Ly, omega, mean, sampler):
    s0 = inputs.random_state(9, Ly, Lx, mean, seed=Lx + 3 * Ly, hot=3, hot_value=900)
    check(B, dict(lattice=3, Lx=Lx, Ly=Ly, omega_eff=omega, seed=11, replica=2, sampler=sampler), s0, 5, 2)


@pytest.mark.parametrize("theta", [0.1, 1.0 / 3.0, 0.9])
@pytest.mark.parametrize("mean", [61.0, 126.0, 600.0])
def test_d2q9_occupations(B, mean, theta):
    s0 = inputs.random_state(9, 7, 19, mean, seed=int(mean), hot=2, hot_value=7000)
    check(B, dict(lattice=3, Lx=19, Ly=7, omega_eff=0.8, theta=theta, seed=13), s0, 4, 2)


@pytest.mark.parametrize("kernel", [6, 7])
@pytest.mark.parametrize("lattice,Lx,Ly", [(1, 8, 1), (1, 4096, 1), (1, 264 * 8, 1), (2, 8, 5), (2, 256, 6), (2, 264, 9),
                                           (2, 2056, 3), (3, 128, 6), (3, 132, 5), (3, 4, 7)])
def test_staged_warp_runs(B, kernel, lattice, Lx, Ly):
    """Ordinary nodes, and vectors whose first, last, several or all nodes hold 64 and more."""
    q = Q[lattice]
    s0 = inputs.random_state(q, Ly, Lx, 7.0, seed=Lx + Ly)
    flat = s0.reshape(q, -1)
    n = flat.shape[1]
    for k, v in ((0, 64), (7, 63), (n - 1, 200), (n // 2, 128)):
        flat[k % q, k] = v
    flat[q - 1, n // 3:n // 3 + 9] = 70
    for omega in (1.7, 0.6):
        check(B, dict(lattice=lattice, Lx=Lx, Ly=Ly, omega_eff=omega, seed=3, replica=4), s0, 7, kernel)


@pytest.mark.parametrize("kernel", [6, 7])
@pytest.mark.parametrize("lattice,mean,omega", [(1, 26.0, 1.6), (2, 20.0, 1.5), (2, 30.0, 1.85), (3, 10.0, 1.5), (3, 14.0, 1.9)])
def test_staged_warp_with_many_slow_nodes(B, kernel, lattice, mean, omega):
    """Means at which a tenth of the nodes and more leave the fast collision."""
    Lx, Ly = (2600 if lattice == 1 else 200), (1 if lattice == 1 else 40)
    s0 = inputs.random_state(Q[lattice], Ly, Lx, mean, seed=int(mean))
    check(B, dict(lattice=lattice, Lx=Lx, Ly=Ly, omega_eff=omega, seed=5), s0, 8, kernel)


@pytest.mark.parametrize("lattice,Lx,Ly", [(2, 560, 557), (2, 640, 487), (2, 644, 487), (1, 311296, 1), (1, 311312, 1),
                                           (2, 1280, 1217)])
def test_default_choice(B, lattice, Lx, Ly):
    s0 = inputs.random_state(Q[lattice], Ly, Lx, 9.0, seed=Lx)
    check(B, dict(lattice=lattice, Lx=Lx, Ly=Ly, omega_eff=1.8, seed=7), s0, 2, -1)
