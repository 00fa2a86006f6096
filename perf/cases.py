"""The work that is measured: what a user of the lattice gas has it do, through the Python
binding of the C ABI (paper_2203_01380_gb300/binding.py).

Every case is a dict of plain values.  Its "kind" names the entry points:

  steps     one lattice (Lattice): T time steps, observables, the state into a device tensor;
            with "init" the pass starts from the Poisson initial state, with "host" the state
            comes from a host array and goes back to one (checkpoint and resume)
  record    D1Q3 rings with the state and the amplitude after every step (Batch.run_record)
  batch     D1Q3 rings of uneven length, occupation and omega_eff (Batch.run), every ring's
            final state, mass and amplitude
  ensemble  equal D1Q3 rings with replica statistics at every step (Batch.ensemble)
  serve     D2Q5 requests of uneven size and length through one Server, with final states
  lb        the lattice Boltzmann comparator (LB) in double precision

Sizes, occupations and omega_eff are those of the repository's workloads
(paper_2203_01380_gb300/inputs.py) with fewer steps, and of its smoke run and tests.
"""
import math

import numpy as np
import torch

from paper_2203_01380_gb300 import binding as B
from paper_2203_01380_gb300 import inputs as I

VELOCITIES = {B.D1Q3: 3, B.D2Q5: 5, B.D2Q9: 9}


def listed():
    return [
        # a short ring followed one step per call (the D1Q3 ring workload, driven from a
        # user's own loop): the smallest call, all latency
        dict(name="ring_one_step", kind="steps", lattice=B.D1Q3, Lx=256, Ly=1, n0=30.0, amp=10.0, omega_eff=1.5, T=1,
             modes=1, init=False, host=True),
        # the D1Q3 ring workload itself: 2000 steps with the state and A^LG after every step
        dict(name="ring_record", kind="record", rings=1, L_min=256, L_max=256, n0_min=30.0, n0_max=30.0, amp=10.0,
             omega_min=1.5, omega_max=1.5, T=2000),
        # a small lattice at low occupation (the smoke run's), resumed from a host state,
        # advanced and saved again
        dict(name="small_resume", kind="steps", lattice=B.D2Q5, Lx=96, Ly=40, n0=12.0, amp=8.0, omega_eff=1.6, T=100,
             modes=2, init=False, host=True),
        # the decay-rate sweep, 1024^2 at 50 per velocity: under-relaxed (no flip, half of the
        # particles redistributed) and strongly over-relaxed (flip, a tenth redistributed)
        dict(name="sweep_under", kind="steps", lattice=B.D2Q5, Lx=1024, Ly=1024, n0=50.0, amp=20.0, omega_eff=0.5,
             T=100, modes=1, init=False, host=False),
        dict(name="sweep_over", kind="steps", lattice=B.D2Q5, Lx=1024, Ly=1024, n0=50.0, amp=20.0, omega_eff=1.9,
             T=100, modes=1, init=False, host=False),
        # odd extents at the highest occupations a request may ask for
        dict(name="odd_dense", kind="steps", lattice=B.D2Q5, Lx=1501, Ly=777, n0=100.0, amp=0.0, omega_eff=1.5, T=50,
             modes=1, init=False, host=False),
        # the structure-factor workload, 16384^2 at 10 per velocity: initial state, steps, S(k)
        dict(name="large_d2q5", kind="steps", lattice=B.D2Q5, Lx=16384, Ly=16384, n0=10.0, amp=0.0, omega_eff=1.8,
             T=50, modes=64, init=True, host=False),
        # the same lattice with nine velocities
        dict(name="large_d2q9", kind="steps", lattice=B.D2Q9, Lx=16384, Ly=16384, n0=10.0, amp=0.0, omega_eff=1.8,
             T=10, modes=64, init=False, host=False),
        # the replica batch: rings of 64 to 8192 nodes, 5 to 200 per velocity, both sides of
        # omega_eff = 1
        dict(name="batch_rings", kind="batch", rings=2048, L_min=64, L_max=8192, n0_min=5.0, n0_max=200.0, amp=0.0,
             omega_min=0.2, omega_max=1.95, T=2000),
        # replica averages of the decaying sine (Sec. V): 512 rings of 320 nodes
        dict(name="ensemble", kind="ensemble", rings=512, L=320, n0=100.0 / 3.0, amp=100.0, omega_eff=1.5, T=2000),
        # a burst of requests served together
        dict(name="serve_burst", kind="serve", requests=24, side_min=64, side_max=1024, steps_min=100, steps_max=1000,
             n0_min=5.0, n0_max=100.0, omega_eff=1.5),
        # the comparator on the sweep's lattice, the sweep's 1000 steps
        dict(name="comparator", kind="lb", lattice=B.D2Q5, Lx=1024, Ly=1024, n0=50.0, amp=20.0, omega_eff=1.8,
             T=1000, modes=1),
    ]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _extent(rng, lo, hi):
    """Log-uniform; a third of the extents a multiple of 8 (vector rows), the others any."""
    n = int(_log_uniform(rng, lo, hi))
    return max(lo, n // 8 * 8) if rng.random() < 1.0 / 3.0 else n


def draw(rng):
    kind = rng.choice(["steps", "steps", "steps", "record", "batch", "ensemble", "serve", "lb"])
    omega = round(rng.uniform(0.2, 1.95), 3)
    n0 = round(_log_uniform(rng, 5.0, 100.0), 2)
    if kind == "steps":
        lattice = rng.choice([B.D1Q3, B.D2Q5, B.D2Q5, B.D2Q9])
        if lattice == B.D1Q3:
            Lx, Ly = _extent(rng, 64, 1 << 22), 1
        else:
            Lx, Ly = _extent(rng, 40, 8192), _extent(rng, 40, 8192)
        T = max(1, min(int(_log_uniform(rng, 1, 500)), (1 << 31) // (Lx * Ly * (2 if lattice == B.D2Q9 else 1))))
        # a sine has one Poisson table per phase: lattices up to the workloads' side
        amp = round(rng.choice([0.0, 0.5]) * n0, 2) if Lx <= 16384 else 0.0
        return dict(kind=kind, lattice=lattice, Lx=Lx, Ly=Ly, n0=n0, amp=amp,
                    omega_eff=omega, T=T, modes=rng.choice([1, 2, 16]), init=rng.random() < 0.3,
                    host=Lx * Ly < (1 << 18) and rng.random() < 0.5)
    if kind in ("record", "batch"):
        rings = int(_log_uniform(rng, 1, 16 if kind == "record" else 1024))
        lo = _extent(rng, 64, 1024)
        hi = max(lo, _extent(rng, 64, 1024 if kind == "record" else 8192))
        T = int(_log_uniform(rng, 50, 1000 if kind == "record" else 2000))
        return dict(kind=kind, rings=rings, L_min=lo, L_max=hi, n0_min=5.0, n0_max=max(10.0, 2.0 * n0), amp=0.0,
                    omega_min=min(0.2, omega), omega_max=max(0.5, omega), T=T)
    if kind == "ensemble":
        return dict(kind=kind, rings=int(_log_uniform(rng, 2, 1024)), L=_extent(rng, 64, 1024), n0=n0,
                    amp=round(0.5 * n0, 2), omega_eff=omega, T=int(_log_uniform(rng, 50, 1000)))
    if kind == "serve":
        return dict(kind=kind, requests=rng.randint(1, 24), side_min=64, side_max=_extent(rng, 65, 1024), steps_min=100,
                    steps_max=int(_log_uniform(rng, 101, 1000)), n0_min=5.0, n0_max=max(10.0, n0), omega_eff=omega)
    lattice = rng.choice([B.D1Q3, B.D2Q5, B.D2Q5, B.D2Q9])
    if lattice == B.D1Q3:
        Lx, Ly = _extent(rng, 64, 1 << 20), 1
    else:
        Lx, Ly = _extent(rng, 40, 1500), _extent(rng, 40, 1500)
    return dict(kind=kind, lattice=lattice, Lx=Lx, Ly=Ly, n0=n0, amp=round(0.5 * n0, 2), omega_eff=omega,
                T=int(_log_uniform(rng, 10, 500)), modes=1)


def _lattice_args(case, seed):
    return dict(lattice=case["lattice"], Lx=case["Lx"], Ly=case["Ly"], n0=case["n0"], amp=case["amp"],
                mode_mx=1 if case["amp"] else 0, init_weighted=0, omega_eff=case["omega_eff"], seed=seed)


def _modes(case):
    """Axis modes as the workloads ask for: along x, and one along y where several are wanted."""
    n = min(case["modes"], case["Lx"] // 2 - 1)
    m = [(k, 0) for k in range(1, n + 1)]
    if case["lattice"] != B.D1Q3 and 1 < n < 64:
        m[-1] = (0, 1)
    return m


# The rings of a batch and the requests of a burst (extents, occupations, omega_eff, steps)
# are drawn once for the case; a seed changes their random streams.
def _rings(case, seed):
    reps = I.batch_replicas(case["rings"], L_min=case["L_min"], L_max=case["L_max"],
                            n0_range=(case["n0_min"], case["n0_max"]), omega_range=(case["omega_min"], case["omega_max"]))
    reps[0]["Lx"] = case["L_max"]  # the longest ring of the range is always there
    sine = dict(amp=case["amp"], mode_mx=1) if case["amp"] else {}
    return [{**r, "seed": seed, **sine} for r in reps]


def _requests(case, seed):
    reqs = I.serve_requests(case["requests"], side_range=(case["side_min"], case["side_max"]),
                            steps_range=(case["steps_min"], case["steps_max"]),
                            n0_range=(case["n0_min"], case["n0_max"]), omega_eff=case["omega_eff"])
    return [dict(r, seed=seed) for r in reqs]


def prepare(case, seed):
    kind, T = case["kind"], case.get("T")
    if kind == "steps":
        lat = B.Lattice(**_lattice_args(case, seed))
        s = dict(kind=kind, T=T, lat=lat, modes=_modes(case), init=case["init"], source=None, out=None)
        if not case["init"]:
            lat.init()
        if not case["host"]:
            # the occupations' 16-bit words (all below 2^15 here)
            s["out"] = torch.empty(lat.shape, dtype=torch.int16, device="cuda")
        elif not case["init"] and T > 1:
            s["source"] = lat.get_state()[0]
        return s
    if kind in ("record", "batch"):
        bat = B.Batch(_rings(case, seed))
        bat.init()
        return dict(kind=kind, T=T, bat=bat)
    if kind == "ensemble":
        one = dict(lattice=B.D1Q3, Lx=case["L"], n0=case["n0"], amp=case["amp"], mode_mx=1, init_weighted=1,
                   omega_eff=case["omega_eff"], seed=seed)
        bat = B.Batch([dict(one, replica=r) for r in range(case["rings"])])
        bat.init()
        return dict(kind=kind, T=T, bat=bat)
    if kind == "serve":
        return dict(kind=kind, srv=B.Server(seed, 1 << 30, max_slots=256, quantum=32), reqs=_requests(case, seed))
    oj, om = B.lb_rates(case["omega_eff"])
    lb = B.LB(omega_j=oj, omega=om, **_comparator_args(case, seed))
    lb.init()
    return dict(kind=kind, T=T, lb=lb, modes=_modes(case))


def _comparator_args(case, seed):
    # the comparator draws nothing: another seed is another mean density
    return dict(_lattice_args(case, 0), n0=case["n0"] * (1.0 + (seed % 1009) / 10090.0))


def run(s):
    kind, T = s["kind"], s.get("T")
    if kind == "steps":
        lat = s["lat"]
        if s["init"]:
            lat.init()
        elif s["source"] is not None:
            lat.set_state(s["source"])
        lat.step(T)
        o = lat.observables(s["modes"])
        if s["out"] is not None:
            state = s["out"]
            lat.get_state_device(state.data_ptr(), state.numel())
        else:
            state = lat.get_state()[0].view(np.int16)
        return [state, o["mass"], o["re"] + 1j * o["im"], o["amp"], o["Sk"]]
    if kind == "record":
        amp, states = s["bat"].run_record(T)
        return [amp, np.concatenate([x.reshape(-1) for x in states]).view(np.int16)]
    if kind == "batch":
        bat = s["bat"]
        bat.run(T)
        mass, amp = bat.observables()
        return [np.concatenate([bat.get_state(i)[0].reshape(-1) for i in range(bat.n)]).view(np.int16),
                mass.view(np.int64), amp]
    if kind == "ensemble":
        stats = s["bat"].ensemble(T)
        mass, amp = s["bat"].observables()
        return [stats, mass.view(np.int64), amp]
    if kind == "serve":
        srv = s["srv"]
        for i, r in enumerate(s["reqs"]):
            srv.submit(i, r["steps"], want_state=True, **{k: v for k, v in r.items() if k not in ("arrive", "steps")})
        srv.wait_idle()
        done = sorted(srv.poll(), key=lambda d: d["id"])
        return [np.concatenate([d["state"].reshape(-1) for d in done]).view(np.int16)] + \
               [np.array([d[k] for d in done]) for k in ("status", "t", "mass", "amp", "Sk")]
    lb = s["lb"]
    lb.step(T)
    o = lb.observables(s["modes"])
    return [lb.get_state()[0], o["mass"], o["re"] + 1j * o["im"], o["amp"]]


def _node_work(lattice, n0, omega_eff):
    """Integer operations of one node update: its Philox4x32-10 words (ten rounds of two wide
    products and four xors per four words) and about six operations per draw and direction
    count.  One word per thinning, rest share and direction group of 32; occupations and
    removals are counted in chunks of 63."""
    Q = VELOCITIES[lattice]
    share = omega_eff if omega_eff <= 1.0 else 2.0 - omega_eff
    removed = share * Q * n0
    rest = {B.D1Q3: 2.0 / 3.0, B.D2Q5: 1.0 / 3.0, B.D2Q9: 4.0 / 9.0}[lattice]
    groups = max(1.0, removed * (1.0 - rest) / 32.0) * (1 if lattice == B.D1Q3 else 2)
    words = Q * max(1.0, n0 / 63.0) + max(1.0, removed / 63.0) + groups
    return words / 4.0 * 60.0 + words * 6.0


def work(case):
    """Bytes: the state read once and written once per pass, and what comes back with it;
    flops: the integer operations of the node updates (comparator: its double-precision ones)."""
    kind = case["kind"]
    if kind in ("steps", "lb"):
        nodes, Q, T = case["Lx"] * case["Ly"], VELOCITIES[case["lattice"]], case["T"]
        if kind == "lb":
            return {"bytes": 16.0 * Q * nodes, "flops": float({3: 14, 5: 24, 9: 42}[Q]) * nodes * T}
        return {"bytes": 4.0 * Q * nodes, "flops": nodes * T * _node_work(case["lattice"], case["n0"], case["omega_eff"])}
    if kind == "serve":
        lat = [(r["Lx"] * r["Ly"], r["steps"], r["n0"]) for r in _requests(case, 0)]
        return {"bytes": sum(20.0 * n for n, _, _ in lat),
                "flops": sum(n * t * _node_work(B.D2Q5, n0, case["omega_eff"]) for n, t, n0 in lat)}
    T = case["T"]
    if kind == "ensemble":
        nodes = case["rings"] * case["L"]
        return {"bytes": 12.0 * nodes + 48.0 * (T + 1),
                "flops": nodes * T * _node_work(B.D1Q3, case["n0"], case["omega_eff"])}
    rings = [(r["Lx"], r["n0"], r["omega_eff"]) for r in _rings(case, 0)]
    nodes = sum(L for L, _, _ in rings)
    record = 6.0 * nodes * T + 8.0 * case["rings"] * T if kind == "record" else 0.0
    return {"bytes": 12.0 * nodes + record, "flops": sum(L * T * _node_work(B.D1Q3, n0, om) for L, n0, om in rings)}


_WEIGHTS = {B.D1Q3: ([4 / 6, 1 / 6, 1 / 6], [(0, 0), (1, 0), (-1, 0)]),
            B.D2Q5: ([1 / 3] + [1 / 6] * 4, [(0, 0), (1, 0), (-1, 0), (0, 1), (0, -1)]),
            B.D2Q9: ([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4,
                     [(0, 0), (1, 0), (-1, 0), (0, 1), (0, -1), (1, 1), (-1, -1), (1, -1), (-1, 1)])}


def exact(case, seed):
    """The comparator's outputs from the relaxation equation written per velocity (odd and
    even parts of f - f^0), in torch.  The gas's outputs are integers and functions of them
    that only its own random stream defines: they are compared with the start's."""
    if case["kind"] != "lb":
        return None
    w, v = _WEIGHTS[case["lattice"]]
    Lx, Ly, Q = case["Lx"], case["Ly"], len(w)
    a = _comparator_args(case, seed)
    # rates of the gas's omega_eff: the flip (above 1) over-relaxes the odd moments only
    oj = case["omega_eff"]
    om = oj if oj <= 1.0 else 2.0 - oj
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    x = torch.arange(Lx, dtype=torch.float64, device=dev)
    lam = a["n0"] + a["amp"] * torch.sin(2.0 * math.pi * x / Lx) / Q
    f = lam.expand(Q, Ly, Lx).clone()
    other = [0] + [i + 1 if i % 2 else i - 1 for i in range(1, Q)]
    for _ in range(case["T"]):
        rho = f.sum(0)
        d = [f[i] - w[i] * rho for i in range(Q)]
        f = torch.stack([torch.roll(w[i] * rho + (1.0 - om) * 0.5 * (d[i] + d[other[i]])
                                    + (1.0 - oj) * 0.5 * (d[i] - d[other[i]]), (v[i][1], v[i][0]), (0, 1))
                         for i in range(Q)])
    rho = f.sum(0)
    mass = float(rho.sum())
    C = (rho - rho.mean()).sum(0)
    k = 2.0 * math.pi / Lx
    re, im = float((torch.cos(k * x) * C).sum()), float((torch.sin(k * x) * C).sum())
    return [f, mass, np.array([re + 1j * im]), np.array([im / (Lx * Ly / 2.0)])]
