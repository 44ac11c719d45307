"""The workloads whose speed is tracked, each one pass of a user's program.

A pass is a block of sweeps and the reads that follow it in a simulation: the
series recorded meanwhile, or one measurement.  ``listed`` names the fixed
cases, ``draw`` gives further ones of the same families over the whole range
of sizes, ``prepare`` builds the lattice a program keeps, ``run`` is one pass
through the package's public calls, and ``work`` counts what a pass cannot do
without.  Every output is a whole number (spins, energies, magnetisations,
overlaps, exchange counts), so outputs of two versions agree exactly or not
at all.
"""

import math

import torch

import paper_0704_3573_gb300 as ianus

# Integer operations one update needs (32-bit; 64-lane words are shared by 64
# updates): random bits, local field or state counts, threshold compare.
OPS = {"ea": 3.3, "pt": 3.7, "plain": 3.3, "field": 4.0, "pool": 3.7, "potts": 36.0, "perm": 45.0, "wheel": 16.0}


def _case(name, family, dim, L, samples, replicas, beta, sweeps, every, algo="heatbath", temps=1, beta_last=0.0,
          disorder="pm_j", field=0.0, occupation=1.0, jobs=0):
    """A case; ``every`` is the measurement cadence (0: one measurement after
    the block), and with parallel tempering also the swap cadence."""
    c = dict(family=family, dim=dim, L=L, samples=samples, replicas=replicas, beta=beta, sweeps=sweeps, every=every,
             algo=algo, temps=temps, beta_last=beta_last, disorder=disorder, field=field, occupation=occupation,
             jobs=jobs)
    if name:
        c = dict(name=name, **c)
    return c


def listed():
    return [
        # a notebook's call: a few sweeps of a small lattice, then its observables
        _case("small_L8_64x2", "ea", 3, 8, 64, 2, 1.0, 10, 0),
        # the paper's single system: one L=16 sample on the plain layout, E and M after every sweep
        _case("single_L16", "plain", 3, 16, 1, 1, 1 / 1.1, 1000, 1, algo="metropolis"),
        # a serving chunk: jobs of several sizes and temperatures in the lanes of one pool
        _case("pool_L16_9jobs", "pool", 3, 16, 256, 1, 1.0, 50, 0, jobs=9),
        # a study with four replicas, a side that is no power of two and a part-filled word
        _case("ragged_L20_100x4", "ea", 3, 20, 100, 4, 0.9, 100, 10, algo="metropolis"),
        # the headline: L=64, 256 samples x 2 replicas, E and Q every 10 sweeps
        _case("headline_L64_256x2", "ea", 3, 64, 256, 2, 1.0, 100, 10),
        # the same update on a state larger than the L2 cache
        _case("large_L128_256x2", "ea", 3, 128, 256, 2, 1.0, 10, 10),
        # equilibration by parallel tempering: 32 temperatures in [0.7, 1.6], swaps every 10 sweeps
        _case("tempering_L32_64x2_K32", "pt", 3, 32, 64, 2, 1 / 0.7, 20, 10, algo="metropolis", temps=32,
              beta_last=1 / 1.6),
        # one byte per spin, the layout for users who read and write spins in place
        _case("plain_L64_256x2", "plain", 3, 64, 256, 2, 1.0, 10, 10),
        # q=4 Potts glass
        _case("potts_L32_128x2", "potts", 3, 32, 128, 2, 1.25, 20, 10),
        # glassy Potts model with permutation couplings, at the paper's temperature
        _case("perm_L32_256x2", "perm", 3, 32, 256, 2, 2.4, 20, 10),
        # random-field Ising model
        _case("rfim_L64_256", "field", 3, 64, 256, 1, 0.5, 20, 10, disorder="rfim", field=1.5),
        # the paper's own generator: Parisi-Rapuano wheels
        _case("wheel_L64_256x2", "wheel", 3, 64, 256, 2, 1.0, 2, 2),
    ]


# Most updates a drawn case of a family makes in one pass (those of its
# largest listed case), and the most sites of its lattices.
MOST_UPDATES = {"ea": 1.07e10, "pt": 2.6e9, "plain": 1.3e9, "field": 1.3e9, "pool": 5e7, "potts": 1.6e8,
                "perm": 3.3e8, "wheel": 2.6e8}


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    family = rng.choice(["ea", "ea", "ea", "pt", "plain", "field", "pool", "potts", "perm", "wheel"])
    dim = rng.choice([3, 3, 3, 2])
    if family == "perm":
        dim = rng.choice([2, 3, 3, 4])
    if family == "pool":
        L = 2 * _log_int(rng, 4, 16) if dim == 3 else 2 * _log_int(rng, 16, 128)
        jobs = rng.randint(2, 16)
        return _case(None, "pool", dim, L, 64 * rng.randint(1, 4), 1, rng.uniform(0.5, 2.0), rng.randint(10, 60), 0,
                     jobs=jobs)
    side = {2: (8, 256), 3: (3, 48), 4: (2, 8)}[dim]
    L = 2 * _log_int(rng, *side)
    N = L ** dim
    temps = _log_int(rng, 2, 32) if family == "pt" else 1
    replicas = rng.choice([1, 1, 2, 2, 2, 3, 4])
    if family == "field":
        replicas = rng.choice([1, 1, 2])
    samples = _log_int(rng, 1, 256)
    # not more work than the largest listed case of the family in two sweeps
    while samples > 1 and 2.0 * samples * replicas * temps * N > MOST_UPDATES[family]:
        samples = (samples + 1) // 2
    while L > 4 and 2.0 * samples * replicas * temps * N > MOST_UPDATES[family]:
        L = 2 * (L // 4)
        N = L ** dim
    sweeps = int(min(100, MOST_UPDATES[family] / (samples * replicas * temps * N)))
    sweeps = max(2, int(sweeps * rng.uniform(0.3, 1.0)))
    every = rng.choice([0, 1, 2, 5, 10])
    algo = rng.choice(["metropolis", "heatbath"]) if family not in ("potts", "perm") else "heatbath"
    kw = {}
    if family == "pt":
        every = min(rng.choice([1, 5, 10]), sweeps)
        sweeps -= sweeps % every
        kw = dict(temps=temps, beta_last=rng.uniform(0.4, 0.7))
        beta = rng.uniform(1.0, 1.5)
    elif family == "field":
        kw = rng.choice([dict(disorder="rfim", field=rng.uniform(0.5, 2.0)),
                         dict(disorder="daff", field=rng.uniform(0.5, 2.0), occupation=rng.uniform(0.6, 0.95))])
        beta = rng.uniform(0.4, 1.2)
    elif family in ("potts", "perm"):
        beta = rng.uniform(0.8, 2.4)
    else:
        beta = 1.0 / rng.uniform(0.5, 2.0)
    return _case(None, family, dim, L, samples, replicas, beta, sweeps, every, algo=algo, **kw)


def _lattice(case, seed):
    family = case["family"]
    rows = case["sweeps"] // case["every"] + 1 if case["every"] else 1
    kw = dict(dim=case["dim"], L=case["L"], n_samples=case["samples"], n_replicas=case["replicas"],
              n_temps=case["temps"], seed=0x0704357300000000 + seed, series_capacity=rows)
    if family == "potts":
        return ianus.Lattice(model="potts", **kw)
    if family == "perm":
        return ianus.Lattice(model="potts_perm", **kw)
    if family == "wheel":
        return ianus.Lattice(rng="wheel", **kw)
    if family == "plain":
        return ianus.Lattice(layout="i8", **kw)
    if family == "field":
        return ianus.Lattice(disorder=case["disorder"], field=case["field"], occupation=case["occupation"], **kw)
    return ianus.Lattice(**kw)


def _spin_view(case, lat):
    """The lattice's spins as they stand in its device buffer, without a copy."""
    n = lat.K * lat.R * lat.N
    if case["family"] in ("plain", "wheel"):
        return lat.buffer[: n * lat.S].view(torch.int8)
    if case["family"] in ("potts", "perm"):
        return lat.buffer[: 4 * n * ((lat.S + 3) // 4)].view(torch.int32)
    return lat.buffer[: 8 * n * ((lat.S + 63) // 64)].view(torch.int64)


def prepare(case, seed):
    """The lattice with couplings and spins from the seed, and what a program
    keeps beside it: the temperatures, or the jobs loaded into a pool."""
    lat = _lattice(case, seed)
    beta = case["beta"]
    if case["family"] == "pt":
        K = case["temps"]
        t0, t1 = 1.0 / beta, 1.0 / case["beta_last"]
        beta = [1.0 / (t0 + (t1 - t0) * k / (K - 1)) for k in range(K)]
    if case["family"] == "pool":
        # jobs of 1 to 64 samples, Metropolis or heat bath, temperatures around
        # the case's, first fit into the groups as the server places them
        groups = case["samples"] // 64
        free = [0] * groups
        for j in range(case["jobs"]):
            n = 1 + (j * 37 + 20) % 64 if j % 3 else 64
            spot = [g for g in range(groups) if free[g] + n <= 64]
            if not spot:
                continue
            algo = ianus.METROPOLIS if j % 2 else ianus.HEATBATH
            lat.segment_load(spot[0], free[spot[0]], n, 1000003 * seed + j, algo, beta * (0.7 + 0.1 * (j % 7)),
                             1 << 40)
            free[spot[0]] += n
    return dict(case=case, lat=lat, beta=beta, spins=_spin_view(case, lat))


def run(state):
    """One block of sweeps and the reads that follow it."""
    case, lat = state["case"], state["lat"]
    if case["family"] == "pool":
        lat.sweep_segments(case["sweeps"])
        E, M, _ = lat.measure(overlap=False)
        return dict(spins=state["spins"], E=E, M=M)
    if case["family"] == "pt":
        lat.sweep_pt(case["algo"], state["beta"], case["sweeps"], case["every"], case["every"])
        slots, accepted, _ = lat.pt_state()
        sweeps, E, M, Q = lat.series(clear=True)
        return dict(spins=state["spins"], slots=slots, accepted=accepted, E=E, M=M, Q=Q)
    lat.sweep(case["algo"], state["beta"], case["sweeps"], case["every"])
    if case["every"]:
        sweeps, E, M, Q = lat.series(clear=True)
    else:
        E, M, Q = lat.measure()
    return dict(spins=state["spins"], E=E, M=M, Q=Q)


def work(case):
    """Bytes: the state read and written once, the disorder read once, the
    observables written.  Operations: those of the updates."""
    family, N = case["family"], case["L"] ** case["dim"]
    S, slots = case["samples"], case["replicas"] * case["temps"]
    if family in ("plain", "wheel"):
        per_sample, pad = N, S
    elif family in ("potts", "perm"):
        per_sample, pad = N, 4 * ((S + 3) // 4)
    else:
        per_sample, pad = N / 8, 64 * ((S + 63) // 64)
    spins = pad * slots * per_sample
    disorder = pad * case["dim"] * per_sample
    if family == "field":
        disorder += pad * per_sample * (2 if case["disorder"] == "daff" else 1)
    if family == "wheel":  # per row and colour the ring of 64 numbers, read and written
        disorder += 2 * S * slots * 2 * 64 * 4 * (N // case["L"])
    every = case["every"]
    rows = case["sweeps"] // every if every else 1
    mq = 4 if family in ("potts", "perm") else 2 if family == "field" else 1
    observables = rows * 8 * (S * slots * (1 + mq) + (S * case["temps"] if case["replicas"] > 1 else 0))
    return {"bytes": 2 * spins + disorder + observables, "flops": OPS[family] * S * slots * N * case["sweeps"]}
