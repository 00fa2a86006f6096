"""The staged warp step's collision of two neighbouring nodes at once, against the oracle: in a
sparse lattice some even nodes, some odd ones and some pairs hold as many particles as bring
the removed and the moving ones to the limits of the fast collision (63 and 32) and beyond,
and occupations to the last table row (63) and beyond, in every position of a vector."""
import numpy as np
import pytest

import oracle as O
from paper_2203_01380_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    from paper_2203_01380_gb300 import binding
    return binding


@pytest.mark.parametrize("lattice,Lx,Ly", [(1, 40, 1), (1, 2088, 1), (2, 8, 5), (2, 264, 6), (2, 44, 9), (3, 264, 6), (3, 44, 9)])
@pytest.mark.parametrize("omega", [0.95, 0.5, 1.3])
@pytest.mark.parametrize("kernel", [6, 7])
def test_pairs_at_the_limits(B, lattice, Lx, Ly, omega, kernel):
    Q = {1: 3, 2: 5, 3: 9}[lattice]
    s0 = inputs.random_state(Q, Ly, Lx, 0.5, seed=Lx + lattice)
    rng = np.random.default_rng(Lx * 5 + Q)
    nodes = s0.reshape(Q, -1)
    # every position of a vector once: alone (even, odd) or with its partner
    for k in range(0, nodes.shape[1] - 1, 5):
        for x in (k, k + 1) if k % 3 == 0 else (k,):
            total = int(rng.integers(28, 80) / min(omega, 2.0 - omega))
            share = rng.multinomial(total, np.ones(Q) / Q)
            share[rng.integers(Q)] = rng.choice([62, 63, 64]) if k % 4 == 0 else share[0]
            nodes[:, x] = share
    cfg = dict(lattice=lattice, Lx=Lx, Ly=Ly, omega_eff=omega, seed=31, replica=4)
    with B.Lattice(**cfg) as lat:
        lat.set_state(s0, 3)
        lat.set_step_kernel(kernel)
        lat.step(1)
        one, _ = lat.get_state()
        lat.step(3)
        got, t = lat.get_state()
    ref = O.Lattice(**cfg)
    assert np.array_equal(one, ref.run(s0, 3, 1))
    assert t == 7 and np.array_equal(got, ref.run(s0, 3, 4))
