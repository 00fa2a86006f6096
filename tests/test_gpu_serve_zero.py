"""Requests of no steps, whose result is the initial state: their state takes part in no round, so
its copy to the caller has to wait for the kernel that writes it.  Alone on an idle server, beside a
request that runs, and on memory that an earlier request of other occupations has left."""
import time

import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu

SEED = 9


def request(i, Lx, Ly, steps, n0):
    return dict(lattice=2, Lx=Lx, Ly=Ly, n0=n0, amp=0.0, omega_eff=1.5, seed=SEED, replica=i, steps=steps)


def want(r):
    return O.Lattice(**{k: v for k, v in r.items() if k != "steps"}).init()


@pytest.mark.parametrize("busy", [False, True])
def test_no_steps(busy):
    from paper_2203_01380_gb300 import binding as B

    with B.Server(SEED, 1 << 29, max_slots=16, quantum=8) as srv:
        if busy:
            srv.submit(100, want_state=False, **request(100, 1000, 900, 400, 60.0))
            time.sleep(0.005)
        for i in range(4):
            r = request(i, 1501 - 2 * i, 1300, 0, (40.0, 5.0, 90.0, 10.0)[i])
            srv.submit(i, want_state=True, **r)
            got = []
            while not got:
                got = [d for d in srv.poll() if d["id"] == i]
            s = want(r)
            assert got[0]["status"] == 0 and got[0]["t"] == 0 and got[0]["mass"] == int(s.sum(dtype=np.int64))
            assert np.array_equal(got[0]["state"], s), i
        srv.wait_idle(300)
