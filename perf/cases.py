"""What the performance of this framework is measured on.

A case is a simulation that a user of the library runs through the Python
binding: a population (with the options of its description), a batch of
independent replicates, a sweep of served jobs, or a spatial community.  One
pass advances it by the case's generations and reads back what such a program
records: the statistics of every generation formed, and, where the program
looks at individuals too, the records or the survivor list of the last one.

Every pass continues from where the last one stopped, as a long simulation
does, so a pass on a state is reproducible from the seed and the number of
passes before it.  Sizes and parameters are those of this repository's own
workloads (N, L, mutation rate, resource, map, weights, deviations, torus).
"""
from __future__ import annotations

import math
from types import SimpleNamespace

import numpy as np

from paper_1603_09255_gb300 import spegg

N_BINS = 4096
LOCI = (32, 64, 128, 256)


# ------------------------------------------------------------------ cases
def _pop(name, n, n_loci, gens, option="none", read="stats", locus=False):
    c = {"kind": "population", "n": n, "n_loci": n_loci, "gens": gens, "option": option, "read": read,
         "locus": locus}
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # an interactive program that looks at every generation: one call forms
        # one small generation, so the launches and the read-back count
        _pop("one-generation-1e3", 1_000, 64, 1),
        # the single-species run of the paper's size: 10,000 x 32 loci, 100
        # generations in one call, its individuals read at the end
        _pop("single-1e4", 10_000, 32, 100, read="records"),
        # a middling population of an odd size with a drawn growth rate of the
        # resource and the allele frequencies of every locus recorded
        _pop("frequencies-99991", 99_991, 64, 100, option="beverton-holt", read="records", locus=True),
        # the headline run: a consumer on a logistic resource, 10^6 x 128 loci,
        # 1,000 generations
        _pop("consumer-1e6", 1_000_000, 128, 1_000, option="logistic", read="records"),
        # the largest population of the served mix, whose parents come from HBM
        _pop("large-2e6", 1_999_993, 256, 100, read="survivors"),
        # the options of a population's description, each on the consumer's size
        # or an odd one: linkage map, parent weights, dominance, and the
        # paper's continuous allelic values
        _pop("map-1e6", 1_000_000, 128, 64, option="map", read="survivors"),
        _pop("weights-1e6", 1_000_000, 128, 128, option="weights", read="survivors"),
        _pop("dominance-300007", 300_007, 128, 128, option="dominance", read="survivors"),
        _pop("continuous-1e6", 1_000_000, 128, 32, option="continuous", read="survivors"),
        # independent replicates of different sizes, loci and selection advanced
        # together, every replicate's trajectory read at the end
        {"name": "replicates-256", "kind": "batch", "count": 256, "n_min": 1_000, "n_max": 200_000, "gens": 200,
         "mix": 12345},
        # a parameter sweep submitted to the server and drained
        {"name": "served-24", "kind": "served", "count": 24, "n_min": 1_000, "n_max": 2_000_000, "gen_min": 100,
         "gen_max": 400, "mix": 2024},
        # three species on a 64 x 64 torus, 10^7 individuals, 256 loci
        {"name": "torus-64x64", "kind": "space", "X": 64, "Y": 64, "n0": 814, "n_loci": 256, "gens": 64},
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["population"] * 7 + ["batch", "served", "space"])
    if kind == "batch":
        n_max = _log_uniform(rng, 4_000, 200_000)
        return {"kind": kind, "count": _log_uniform(rng, 8, 256), "n_min": 1_000, "n_max": n_max,
                "gens": rng.randint(20, 200), "mix": rng.randrange(1 << 30)}
    if kind == "served":
        n_max = _log_uniform(rng, 10_000, 500_000)
        return {"kind": kind, "count": rng.randint(4, 24), "n_min": 1_000, "n_max": n_max, "gen_min": 50,
                "gen_max": rng.randint(100, 400), "mix": rng.randrange(1 << 30)}
    if kind == "space":
        return {"kind": kind, "X": rng.randint(8, 64), "Y": rng.randint(8, 64), "n0": _log_uniform(rng, 50, 814),
                "n_loci": rng.choice(LOCI), "gens": rng.randint(1, 64)}
    option = rng.choice(["none", "none", "logistic", "logistic", "beverton-holt", "map", "weights", "dominance",
                         "continuous"])
    n_loci = rng.choice(LOCI)
    n = _log_uniform(rng, 1_000, 1_000_000 if option in ("map", "continuous") else 2_000_000)
    # at most the work of the listed cases: bytes of a pass below the consumer's
    most = 2e10 / (_bytes_per_offspring(n_loci, option) * n)
    gens = max(1, min(_log_uniform(rng, 1, 1_000), int(most)))
    read = rng.choice(["stats", "survivors", "records"])
    if read == "records" and 8 * n * n_loci > (1 << 30):
        read = "survivors"
    if option == "continuous" and read == "records":
        read = "survivors"
    return _pop(None, n, n_loci, gens, option, read, locus=option == "logistic" and rng.random() < 0.3)


# ------------------------------------------------------------------ inputs
def _effects(n_loci, rng, sd=0.1):
    """Effects N(0, sd) in Q8."""
    return np.clip(np.rint(rng.normal(0.0, sd, n_loci) * 256.0), -32768, 32767).astype(np.int16)


def _bins(raw_min, raw_max):
    shift = 0
    while ((raw_max - raw_min) >> shift) >= N_BINS:
        shift += 1
    return -raw_min, shift


def _trait(bias, shift):
    return (np.arange(N_BINS) * float(1 << shift) - bias + ((1 << shift) - 1.0) / 2.0) / 512.0


def _stabilizing(z, s, theta=0.0):
    """exp(-s (z - theta)^2) as thresholds of 2^32."""
    w = np.exp(-s * (z - theta) ** 2)
    t = np.minimum(np.floor(w * 4294967296.0), 4294967294.0).astype(np.uint64)
    t[w >= 1.0] = 0xFFFFFFFF
    return t.astype(np.uint32)


def _weights(z, slope):
    return (np.floor(65536.0 * (1.0 + np.tanh(slope * z))) + 1.0).astype(np.uint32)


def _workload(n, n_loci, seed, replicate, rng, mu, s=0.5, option="none"):
    e = _effects(n_loci, rng)
    e64 = e.astype(np.int64)
    d = None
    if option == "dominance":
        d = _effects(n_loci, rng)
        v = np.stack([np.zeros_like(e64), e64 + d, 2 * e64])
        bias, shift = _bins(int(v.min(axis=0).sum()), int(v.max(axis=0).sum()))
    elif option == "continuous":
        span = 2 * int(np.abs(e64).sum()) + 4096 * 4
        bias, shift = _bins(-span, span)
    else:
        bias, shift = _bins(2 * int(np.minimum(e64, 0).sum()), 2 * int(np.maximum(e64, 0).sum()))
    z = _trait(bias, shift)
    w = SimpleNamespace(n=n, n_loci=n_loci, seed=seed, replicate=replicate, effects=e, bias=bias, shift=shift,
                        surv_table=_stabilizing(z, s), mu=mu, p0_q32=0x80000000, init_genotypes=None, dominance=d,
                        has_ecology=False)
    if option in ("logistic", "beverton-holt", "map", "weights", "dominance"):  # the consumer's resource, K = 10 N
        w.has_ecology = True
        w.eco_r, w.eco_K, w.eco_R0, w.eco_R_half = 0.5, 10.0 * n, 5.0 * n, 1.0 * n
        w.attack = np.clip(np.rint((1.0 + 0.5 * np.tanh(z)) * 65536.0), 0, 2 ** 32 - 1).astype(np.uint32)
        w.eco_model, w.eco_r_sd = 0, 0.0
    if option == "beverton-holt":
        w.eco_r, w.eco_model, w.eco_r_sd = 2.0, 1, 0.2
    if option == "map":  # four chromosomes of one Morgan
        per = n_loci // 4
        w.map_morgans = np.full(n_loci, 1.0 / (per - 1))
        w.map_morgans[::per] = -1.0
    if option == "weights":
        w.mother_weights, w.father_weights = _weights(z, 1.0), _weights(z, 2.0)
    if option == "continuous":
        w.allele_model, w.mut_sd, w.env_sd, w.mu = 1, 0.05, 0.2, 1e-3
    return w


def _mix(case, seed, loci, s_max=0.5, mu=1e-5):
    """Workloads of a batch or a sweep: sizes, loci and selection from the
    case's mix, effects and random streams from the seed."""
    sizes, rng = np.random.default_rng(case["mix"]), np.random.default_rng(seed)
    out = []
    for r in range(case["count"]):
        n = int(round(math.exp(sizes.uniform(math.log(case["n_min"]), math.log(case["n_max"])))))
        n_loci, s = int(sizes.choice(loci)), float(sizes.uniform(0.0, s_max))
        gens = int(sizes.integers(case["gen_min"], case["gen_max"] + 1)) if "gen_min" in case else case["gens"]
        out.append((n, n_loci, s, gens))
    return [(_workload(n, n_loci, seed, r, rng, mu, s), gens) for r, (n, n_loci, s, gens) in enumerate(out)]


def _community(case, seed):
    """Prey, competitor and predator, as in the spatial workload."""
    rng = np.random.default_rng(seed)
    scale = [[0.80, 0.90, 0.82], [0.80, 0.90, 0.82], [0.85, 0.92, 0.85]]
    k = case["n0"] / 814.0  # interactions at the founders' density whatever it is
    species = []
    for q in range(3):
        e = _effects(case["n_loci"], rng)
        e64 = e.astype(np.int64)
        bias, shift = _bins(2 * int(np.minimum(e64, 0).sum()), 2 * int(np.maximum(e64, 0).sum()))
        w = _stabilizing(_trait(bias, shift), 0.3, float(e64.sum()) / 512.0).astype(np.float64)
        tables = np.stack([np.minimum(np.floor(w * a), 4294967294.0) for a in scale[q]]).astype(np.uint32)
        species.append(SimpleNamespace(
            effects=e, tables=tables, bias=bias, shift=shift, mu=1e-5, n0=case["n0"], p0_q32=0x80000000,
            D=int(400000 * k), A=[[1, 1, 3], [1, 1, 3], [0, 0, 1]][q], G=int([1500, 1500, 0][q] * k),
            P=[[0, 0, 0], [0, 0, 0], [1, 1, 0]][q], E=int([0, 0, 500][q] * k),
            C=[[2, 0, 0], [0, 2, 0], [0, 0, 2]][q], beta_q16=int([0.7, 0.7, 0.65][q] * 65536), bmax=2 * case["n0"]))
    return SimpleNamespace(X=case["X"], Y=case["Y"], patches=case["X"] * case["Y"], n_loci=case["n_loci"], seed=seed,
                           disp_q32=int(0.05 * 4294967296.0), species=species)


def prepare(case, seed):
    st = SimpleNamespace(case=case, gen=0)
    if case["kind"] == "population":
        mu = 1e-4 if case["n"] <= 10_000 else 1e-5
        w = _workload(case["n"], case["n_loci"], seed, 0, np.random.default_rng(seed), mu, option=case["option"])
        st.pop = spegg.Population.from_workload(w, stats_capacity=max(case["gens"], 64))
        st.survivors = np.full(case["n"], -1, np.int32)
        if case["locus"]:
            st.pop.set_locus_counts(True)
    elif case["kind"] == "batch":
        st.members = [w for w, _ in _mix(case, seed, (32, 64, 128))]
        st.batch = spegg.Batch(st.members, stats_capacity=max(case["gens"], 64))
    elif case["kind"] == "served":
        st.jobs = _mix(case, seed, (64, 256))
        st.server = spegg.Server(gens_per_tick=16)
    else:
        st.space = spegg.Space(_community(case, seed), stats_capacity=max(case["gens"], 64))
    return st


# -------------------------------------------------------------------- pass
def _fields(stats):
    """The fields of statistics records as plain arrays (whole numbers signed)."""
    out = {}
    for name in stats.dtype.names:
        if name != "pad":
            a = np.ascontiguousarray(stats[name])
            out[name] = a if a.dtype.kind == "f" else a.view("<i%d" % a.dtype.itemsize)
    return out


def run(st):
    case = st.case
    if case["kind"] == "served":
        jobs = [(st.server.submit(w, gens, 0.0), gens) for w, gens in st.jobs]
        st.server.drain()
        return _fields(np.concatenate([st.server.job_stats(j, 1, gens) for j, gens in jobs]))
    first, st.gen = st.gen + 1, st.gen + case["gens"]
    if case["kind"] == "batch":
        st.batch.step(case["gens"])
        return _fields(np.concatenate([st.batch.read_stats(i, first, case["gens"]) for i in range(case["count"])]))
    if case["kind"] == "space":
        st.space.step(case["gens"])
        return {**_fields(st.space.read_stats(first, case["gens"])), "sizes": st.space.sizes()}
    pop = st.pop
    pop.step(case["gens"])
    out = _fields(pop.read_stats(first, case["gens"]))
    if case["locus"]:
        out["locus_counts"] = pop.locus_counts(first, case["gens"]).view(np.int32)
    if case["read"] == "records":
        out["records"] = pop.genotypes().view(np.int32)
    if case["read"] in ("records", "survivors"):  # the list in a buffer for all n, -1 past its end
        alive = pop.survivors()
        st.survivors[:alive.size], st.survivors[alive.size:] = alive, -1
        out["survivors"] = st.survivors
    return out


# -------------------------------------------------------------------- work
def _bytes_per_offspring(n_loci, option="none"):
    """Two parent records read, the child's written, and its survivor index."""
    return 12 + 3 * (4 * n_loci if option == "continuous" else n_loci // 4)


def work(case):
    if case["kind"] == "population":
        b = case["n"] * case["gens"] * _bytes_per_offspring(case["n_loci"], case["option"])
    elif case["kind"] == "space":
        # every individual's record and age read and written once each step
        b = 3 * case["X"] * case["Y"] * case["n0"] * case["gens"] * (case["n_loci"] // 2 + 2)
    else:
        loci = (32, 64, 128) if case["kind"] == "batch" else (64, 256)
        sizes, b = np.random.default_rng(case["mix"]), 0
        for _ in range(case["count"]):
            n = int(round(math.exp(sizes.uniform(math.log(case["n_min"]), math.log(case["n_max"])))))
            n_loci, _ = int(sizes.choice(loci)), sizes.uniform(0.0, 0.5)
            gens = int(sizes.integers(case["gen_min"], case["gen_max"] + 1)) if "gen_min" in case else case["gens"]
            b += n * gens * _bytes_per_offspring(n_loci)
    return {"bytes": b, "flops": 0}


def exact(case, seed):
    """Every output is a whole number or follows from whole numbers by a few
    double operations a generation (the resource R); plain numpy would need
    the whole simulation for it, over 20 seconds for the cases with a resource."""
    return None
