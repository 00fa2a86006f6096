"""Batches of few rings, whose rings are split between the blocks of a cluster: lengths around
the shortest that is split, that leave parts of unlike size, rings too short to be split
beside long ones (down to three nodes), the longest ring, every number of rings per cluster
size; steps beyond several exchanges of the halos and the 64 steps whose words are made
ahead; more rings than clusters, which pull them, the short ones one per block; both samplers and
probabilities that are never or always; a ring that overflows after its beams have crossed the
border of two parts, and one of a block of its own.  States bit for bit; amplitudes as for the
unsplit rings (1e-12 of the sum of magnitudes, 2^-62 fixed point against extended precision)."""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    from paper_2203_01380_gb300 import binding
    return binding


def rings(Ls, **kw):
    return [dict(dict(lattice=1, Lx=L, n0=12.0, amp=3.0, mode_mx=1, omega_eff=1.4, seed=21, replica=i), **kw)
            for i, L in enumerate(Ls)]


CASES = [([256], 90, {}), ([257, 3, 5, 31, 63, 64, 95], 75, {}), ([1000] * 16 + [97], 40, dict(n0=90.0)),
         ([10240], 30, {}), ([4099, 300, 8192], 35, dict(omega_eff=0.6)), ([700] * 50, 25, {}), ([511] * 76, 25, {}),
         ([2500] * 12 + [700] * 40 + list(range(3, 74)), 30, {}), ([2000] * 5 + [130, 255, 256, 77] * 30, 30, dict(sampler=1)),
         ([600, 40], 30, dict(sampler=1)), ([333], 30, dict(omega_eff=2.0)), ([333], 30, dict(omega_eff=1.0, n0=150.0))]


@pytest.mark.parametrize("Ls,T,kw", CASES)
def test_split_rings(B, Ls, T, kw):
    reps = rings(Ls, **kw)
    which = [i for i in range(len(Ls)) if i < 7 or i == len(Ls) - 1]
    with B.Batch(reps) as a, B.Batch(reps) as b:
        a.init()
        amp, states = a.run_record(T, record_mode=2)
        b.init()
        b.run(T)
        for i in which:
            ref = O.Lattice(**reps[i])
            s = ref.init()
            for t in range(T):
                s = ref.step(s, t)
                assert np.array_equal(states[i][t], s), (i, t)
                if t % 7 == 0 or t == T - 1:
                    _, _, _, res = ref.observables(s, [(2, 0)])
                    tol = 1e-12 * res[0]["scale"] / (reps[i]["Lx"] / 2.0)
                    assert abs(amp[i, t] - res[0]["amp"]) <= tol + 1e-300, (i, t)
            assert np.array_equal(a.get_state(i)[0], s) and np.array_equal(b.get_state(i)[0], s)


@pytest.mark.parametrize("L,more", [(300, []), (300, [2500] * 12 + [90] * 120), (200, [2500] * 12 + [90] * 120)])
def test_split_ring_overflows(B, L, more):
    # two beams meet at a crowded node between two parts
    reps = rings([L, L] + more, omega_eff=0.02, theta=0.01, amp=0.0)
    s0 = np.full((3, 1, L), 5, np.uint16)
    s0[0, 0, 100], s0[1, 0, 80], s0[2, 0, 120] = 65400, 48000, 48000
    ref = O.Lattice(**reps[0])
    s, t = s0, 3
    with pytest.raises(OverflowError):
        while t < 60:
            s, t = ref.step(s, t), t + 1
    assert t == 23
    with B.Batch(reps) as bat:
        for record in (True, False):
            bat.init()
            bat.set_state(0, s0, 3)
            with pytest.raises(B.IlgError) as e:
                bat.run_record(50) if record else bat.run(50)
            assert e.value.status == B.ILG_E_OVERFLOW
            got, at = bat.get_state(0)
            assert at == t and np.array_equal(got, s)
            got, at = bat.get_state(1)
            other = O.Lattice(**reps[1])
            assert at == 50 and np.array_equal(got, other.run(other.init(), 0, 50))
