"""The server's shares of a round where they can go wrong: many lattices to a block (more
tables than it holds and more descriptors than it keeps), lattices cut between blocks, both
samplers and probabilities of 0 and 1 in one mix, the densest start, requests that end at
different steps of a round."""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu

SEED = 9


@pytest.fixture(scope="module")
def B():
    from paper_2203_01380_gb300 import binding
    return binding


def serve(B, reqs, quantum, slots=512):
    with B.Server(SEED, 1 << 28, max_slots=slots, quantum=quantum) as srv:
        for i, r in enumerate(reqs):
            srv.submit(i, want_state=True, **r)
        srv.wait_idle(300)
        done = {d["id"]: d for d in srv.poll(4096)}
    assert set(done) == set(range(len(reqs)))
    return done


def check(reqs, done, which):
    for i in which:
        cfg = {k: v for k, v in reqs[i].items() if k != "steps"}
        ref = O.Lattice(**cfg)
        want = ref.run(ref.init(), 0, reqs[i]["steps"])
        assert done[i]["status"] == 0 and done[i]["t"] == reqs[i]["steps"]
        assert np.array_equal(done[i]["state"], want), i
        assert done[i]["mass"] == int(want.sum(dtype=np.int64))


def request(i, Lx, Ly, steps, **kw):
    return dict(dict(lattice=2, Lx=Lx, Ly=Ly, n0=8.0, amp=0.0, omega_eff=1.5, seed=SEED, replica=i, steps=steps), **kw)


@pytest.mark.parametrize("quantum", [1, 5, 64])
def test_many_lattices_to_a_block(B, quantum):
    rng = np.random.default_rng(quantum)
    reqs = [request(i, int(rng.integers(3, 9)), int(rng.integers(3, 9)), int(rng.integers(1, 20)),
                    n0=float(rng.uniform(2, 90)), omega_eff=float(rng.choice([0.4, 1.0, 1.5, 2.0])),
                    theta=float(rng.choice([1.0 / 3.0, 0.5])), sampler=int(i % 7 == 3)) for i in range(260)]
    check(reqs, serve(B, reqs, quantum), range(len(reqs)))


def test_lattices_cut_between_blocks(B):
    """A large lattice, and a middle-sized one of odd rows at other occupations, cut between
    blocks that also hold small ones."""
    reqs = [request(0, 301, 203, 7, n0=70.0), request(1, 45, 33, 13), request(2, 200, 150, 6, n0=5.0, omega_eff=0.8),
            request(3, 3, 3, 20), request(4, 129, 65, 9, n0=100.0, omega_eff=1.0)]
    check(reqs, serve(B, reqs, 8), range(len(reqs)))


def test_densest_start(B):
    """The largest mean a request may have, nearly all of it at rest, beside an ordinary one."""
    reqs = [request(0, 3, 3, 30, n0=700.0, omega_eff=1.0, theta=0.004), request(1, 64, 64, 30)]
    check(reqs, serve(B, reqs, 16), [0, 1])
