"""Initial states of lattices large enough for the guided inversion (one mean per weight
class), against the oracle bit for bit: rows and totals that are and are not a multiple of
four nodes, every velocity set, one to three weight classes, means from nearly nothing to the
largest, and the extent on either side of which the plain inversion runs."""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cfg", [
    dict(lattice=2, Lx=1000, Ly=700, n0=10.0, seed=1),
    dict(lattice=2, Lx=801, Ly=801, n0=50.0, seed=2, replica=3),
    dict(lattice=2, Lx=902, Ly=699, n0=700.0, seed=3),
    dict(lattice=2, Lx=900, Ly=720, n0=90.0, init_weighted=1, theta=0.45, seed=4),
    dict(lattice=2, Lx=900, Ly=700, n0=0.003, seed=5),
    dict(lattice=3, Lx=900, Ly=700, n0=30.0, init_weighted=1, seed=6),
    dict(lattice=3, Lx=901, Ly=703, n0=5.0, seed=7),
    dict(lattice=1, Lx=700001, n0=33.0, init_weighted=1, seed=8),
    dict(lattice=1, Lx=700004, n0=120.0, seed=1 << 40),
    dict(lattice=2, Lx=152, Ly=4095, n0=20.0, seed=10),
    dict(lattice=2, Lx=152, Ly=4096, n0=20.0, seed=10),
])
def test_init_of_large_lattices(cfg):
    from paper_2203_01380_gb300 import binding as B
    with B.Lattice(**cfg) as lat:
        lat.init()
        got, t = lat.get_state()
    assert t == 0 and np.array_equal(got, O.Lattice(**cfg).init())
