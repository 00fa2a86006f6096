"""The comparator's mass and projections where their kernels' blocks end: one column block
and two, one chunk of rows and two, the sides at which a projection takes more blocks or
larger chunks, the longest side whose mass is summed with the columns and one more, and more
modes than travel with the launch; each call twice (the blocks' arrival counters must be back
at zero).  Against extended precision."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

D1Q3, D2Q5, D2Q9 = 1, 2, 3
Q = {D1Q3: 3, D2Q5: 5, D2Q9: 9}


@pytest.fixture(scope="module")
def B():
    from paper_2203_01380_gb300 import binding
    return binding


def expected(f, modes):
    rho = f.astype(np.longdouble).sum(0)
    col, row = rho.sum(0), rho.sum(1)
    mass = col.sum()
    out = []
    for mx, my in modes:
        s, m = (col, mx) if mx else (row, my)
        L = len(s)
        r = (np.arange(L, dtype=np.int64) * m) % L
        ph = 8 * np.arctan(np.longdouble(1)) * r.astype(np.longdouble) / L
        d = s - mass / L
        out.append((float((np.cos(ph) * d).sum()), float((np.sin(ph) * d).sum())))
    return float(mass), np.array(out)


@pytest.mark.parametrize("lattice,Lx,Ly,modes", [
    (D2Q5, 3, 3, [(1, 0), (0, -1)]),
    (D2Q5, 255, 64, [(1, 0), (0, 2), (-3, 0)]),
    (D2Q9, 256, 65, [(1, 0), (0, 1)]),
    (D2Q9, 257, 129, [(k + 1, 0) for k in range(64)]),
    (D2Q5, 40, 300, [((k + 1) if k % 2 else 0, 0 if k % 2 else k + 1) for k in range(65)]),
    (D2Q5, 4096, 7, [(5, 0), (0, 3)]),
    (D2Q5, 4097, 5, [(5, 0), (0, 2)]),
    (D2Q5, 5, 4097, [(2, 0), (0, 7)]),
    (D1Q3, 65536, 1, [(1, 0)]),
    (D1Q3, 65537, 1, [(1, 0), (-4, 0)]),
    (D1Q3, (1 << 20) + 3, 1, [(3, 0)]),
])
def test_sums_match_extended_precision(B, lattice, Lx, Ly, modes):
    rng = np.random.default_rng(Lx * 31 + Ly)
    f = rng.uniform(1.0, 20.0, (Q[lattice], Ly, Lx))
    with B.LB(lattice, Lx, Ly) as lb:
        lb.set_state(f)
        got = [lb.observables(modes) for _ in range(2)]
    mass, want = expected(f, modes)
    # plain sums of Q values, 64 rows and their chunks (rows: one in 256 columns, 8 halvings)
    # on every entry, then compensated sums of products: each rounding is of at most the mass
    roundings = Q[lattice] + 64 + Ly // 64 + Lx // 256 + 8 + 16
    tol = 2.0 * roundings * 2.0**-53 * mass
    for o in got:
        assert abs(o["mass"] - mass) <= tol
        assert np.max(np.abs(o["re"] - want[:, 0])) <= tol
        assert np.max(np.abs(o["im"] - want[:, 1])) <= tol
    for key in ("mass", "re", "im"):
        assert np.array_equal(got[0][key], got[1][key])
