"""Block shapes and records of the batch kernel where they can go wrong: rings shorter than
a warp, of one warp, one node more, and longer than the block; more rings than SMs (the
256-thread blocks); records whose number of states is no multiple of the group they are
written out in, and more than 64 steps (the launch-wide words are made 32 steps at a time);
a recording ring that overflows beside one that does not; two batches with rings of
different length alive at once."""
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


def check_record(B, reps, T, which):
    with B.Batch(reps) as bat:
        bat.init()
        amp, states = bat.run_record(T, record_mode=2)
        final = [bat.get_state(i)[0] for i in which]
    for i, got_final in zip(which, final):
        ref = O.Lattice(**reps[i])
        s = ref.init()
        for t in range(T):
            s = ref.step(s, t)
            assert np.array_equal(states[i][t], s), (i, t)
            if t % 7 == 0 or t == T - 1:
                M, _, _, res = ref.observables(s, [(2, 0)])
                tol = 1e-12 * res[0]["scale"] / (reps[i]["Lx"] / 2.0)
                assert abs(amp[i, t] - res[0]["amp"]) <= tol + 1e-300, (i, t)
        assert np.array_equal(got_final, s)


@pytest.mark.parametrize("L,T", [(3, 9), (31, 8), (32, 7), (33, 16), (161, 70), (256, 3), (257, 9), (1025, 5)])
def test_record_of_one_ring(B, L, T):
    check_record(B, rings([L]), T, [0])


@pytest.mark.parametrize("n0,omega", [(12.0, 1.4), (90.0, 0.8), (30.0, 1.0), (30.0, 2.0)])
def test_record_with_more_rings_than_sms(B, n0, omega):
    Ls = [320] * 150 + [5, 33, 64, 250, 319] * 4
    check_record(B, rings(Ls, n0=n0, omega_eff=omega), 17, [0, 149, 150, 151, 152, 153, 169])


def test_recording_ring_overflows(B):
    reps = rings([100, 100], omega_eff=1.0, theta=0.01, amp=0.0)
    s0 = np.full((3, 1, 100), 5, np.uint16)
    s0[:, 0, 40] = 30000  # 98.5 % of 90000 come to rest at once
    with B.Batch(reps) as bat:
        bat.init()
        bat.set_state(0, s0, 3)
        with pytest.raises(B.IlgError) as e:
            bat.run_record(20)
        assert e.value.status == B.ILG_E_OVERFLOW
        got, t = bat.get_state(0)
        assert t == 3 and np.array_equal(got, s0)
        got, t = bat.get_state(1)
        ref = O.Lattice(**reps[1])
        assert t == 20 and np.array_equal(got, ref.run(ref.init(), 0, 20))


def test_two_batches_of_different_length(B):
    a, b = rings([5000]), rings([1500, 40])
    with B.Batch(a) as x, B.Batch(b) as y:
        for bat, reps in ((x, a), (y, b), (x, a)):
            bat.init()
            bat.run(3)
            ref = O.Lattice(**reps[0])
            assert np.array_equal(bat.get_state(0)[0], ref.run(ref.init(), 0, 3))
