"""Sums and projections at the sizes where their kernels can go wrong: rows of whole and of
ragged vectors, fewer rows than a block's groups and more than one chunk of them, one and
several chunks per mode, more modes than one launch takes, a state that is not aligned for
vector loads, the largest occupations; and the same results call after call (the scratch is
left as it was found)."""
import numpy as np
import pytest

import oracle as O
from paper_2203_01380_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    from paper_2203_01380_gb300 import binding
    return binding


def check(state, obs, modes, Lx, Ly):
    N = state.astype(np.int64).sum(axis=0)
    col, row, M = N.sum(axis=0), N.sum(axis=1), int(N.sum())
    assert obs["mass"] == M
    if obs.get("col") is not None:
        assert np.array_equal(obs["col"], col) and np.array_equal(obs["row"], row)
    for i, (mx, my) in enumerate(modes):
        sums, L, m = (col, Lx, mx) if my == 0 else (row, Ly, my)
        re, im, scale = O.project_exact(sums, L, m, M)
        assert abs(obs["re"][i] - re) <= 1e-12 * scale + 1e-300 and abs(obs["im"][i] - im) <= 1e-12 * scale + 1e-300


@pytest.mark.parametrize("lattice,Lx,Ly", [(2, 8, 3), (2, 264, 7), (2, 256, 9), (2, 40, 4999), (2, 33, 65), (2, 63, 8),
                                           (2, 2051, 17), (3, 72, 130), (3, 31, 33), (1, 8, 1), (1, 65, 1), (1, 4104, 1),
                                           (1, 100003, 1)])
def test_sums_and_projections(B, lattice, Lx, Ly):
    Q = {1: 3, 2: 5, 3: 9}[lattice]
    s0 = inputs.random_state(Q, Ly, Lx, 40.0, seed=Lx + Ly, hot=5, hot_value=65535)
    modes = [(1, 0), (Lx // 3, 0), (-2, 0)] + ([] if lattice == 1 else [(0, 1), (0, Ly - 1)])
    with B.Lattice(lattice, Lx, Ly, omega_eff=1.5, seed=1) as lat:
        lat.set_state(s0)
        first = lat.observables(modes, col_sums=True, row_sums=True)
        again = lat.observables(modes)
        none = lat.observables()
    check(s0, first, modes, Lx, Ly)
    assert none["mass"] == first["mass"]
    for k in ("re", "im", "amp", "Sk"):
        assert np.array_equal(first[k], again[k])


def test_more_modes_than_a_launch_takes(B):
    Lx, Ly = 600, 20
    s0 = inputs.random_state(5, Ly, Lx, 20.0, seed=2)
    modes = [(1 + i % 500, 0) if i % 3 else (0, 1 + i % 19) for i in range(270)]
    with B.Lattice(2, Lx, Ly, omega_eff=1.5, seed=1) as lat:
        lat.set_state(s0)
        check(s0, lat.observables(modes), modes, Lx, Ly)


def test_unaligned_state(B):
    """A caller's state that starts on an odd 16-bit word takes the scalar loads."""
    import torch
    Lx, Ly = 64, 24
    s0 = inputs.random_state(5, Ly, Lx, 20.0, seed=3)
    for off in (0, 1, 8):
        buf = torch.zeros(off + s0.size, dtype=torch.int16, device="cuda")
        buf[off:] = torch.from_numpy(s0.reshape(-1).view(np.int16)).cuda()
        torch.cuda.synchronize()
        modes = [(1, 0), (0, 2)]
        check(s0, B.observables_noalloc(2, Lx, Ly, buf.data_ptr() + 2 * off, modes), modes, Lx, Ly)


@pytest.mark.parametrize("low,high", [(20000, 21000), (65000, 65535)])
def test_products_near_and_beyond_128_bits(B, low, high):
    # L * M just below 2^64 (integer sums) and beyond (double sums), eight phases
    L = 1 << 24
    s0 = np.full((3, 1, L), low, np.uint16)
    s0[:, 0, 1::8] = high
    s0[1, 0, 2::8] = high
    with B.Lattice(1, L, 1, omega_eff=1.5, seed=1) as lat:
        lat.set_state(s0)
        got = lat.observables([(L // 8, 0)])
    S = [3 * low, 3 * high, 2 * low + high] + [3 * low] * 5  # column sums of the phase classes
    M = sum(S) * (L // 8)
    assert got["mass"] == M and (L * M < 2**64) == (low == 20000)
    D = [np.longdouble(L // 8) * (np.longdouble(8 * s - sum(S)) / 8) for s in S]
    ph = [4 * np.arctan(np.longdouble(1)) * c / 4 for c in range(8)]
    re, im = (sum(f(p) * d for p, d in zip(ph, D)) for f in (np.cos, np.sin))
    # the sines and cosines are off by two ulps at most, the sums are rounded once
    tol = 8 * 2.0**-53 * float(sum(abs(d) for d in D))
    assert abs(got["re"][0] - re) <= tol and abs(got["im"][0] - im) <= tol
