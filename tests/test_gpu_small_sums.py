"""The mass and projections of a small lattice in one launch, at the ends of its range (sides of
2048 nodes, 16384 nodes, 32 modes) and beyond, at the least sides, where blocks have no entry,
and at occupations up to 65535: against exact sums (1e-12 of the sum of magnitudes, as for the
two launches) and, bit for bit, against the two launches, which a call that asks for the column
sums takes."""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lattice,Lx,Ly,nmodes", [(1, 3, 1, 1), (1, 2048, 1, 32), (1, 2049, 1, 3), (2, 3, 3, 2), (2, 7, 2048, 5),
                                                  (2, 2048, 8, 33), (2, 128, 128, 32), (2, 129, 128, 3), (3, 8, 2048, 4),
                                                  (3, 61, 57, 9)])
def test_one_launch(lattice, Lx, Ly, nmodes):
    from paper_2203_01380_gb300 import binding as B

    Q = {1: 3, 2: 5, 3: 9}[lattice]
    state = np.random.default_rng(Lx * Ly).integers(0, 65536, (Q, Ly, Lx)).astype(np.uint16)
    modes = [(1 + i % (Lx - 1), 0) if lattice == 1 or i % 2 == 0 else (0, -1 - i % (Ly - 1)) for i in range(nmodes)]
    with B.Lattice(lattice, Lx, Ly, omega_eff=1.5, seed=1) as lat:
        lat.set_state(state)
        got = lat.observables(modes)
        two = lat.observables(modes, col_sums=True)
    N = state.astype(np.int64).sum(axis=0)
    M = int(N.sum())
    assert got["mass"] == M
    for k in ("re", "im", "amp", "Sk"):
        assert np.array_equal(got[k], two[k]), k
    for i, (mx, my) in enumerate(modes):
        sums, L, m = (N.sum(axis=0), Lx, mx) if my == 0 else (N.sum(axis=1), Ly, my)
        re, im, scale = O.project_exact(sums, L, m, M)
        assert abs(got["re"][i] - re) <= 1e-12 * scale + 1e-300 and abs(got["im"][i] - im) <= 1e-12 * scale + 1e-300
