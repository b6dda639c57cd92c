"""The work that programs have this framework do, as timed cases: Metropolis
sweeps of single lattices, batches, multispin ensembles and served jobs, the
exchange of configurations with the host, and the measures, each through the
public entry points of paper_1411_0127_gb300.

A case's inputs (couplings, spins, generator streams) are made inside the
library from seeds, as every program of this framework does; a pass continues
the trajectory where the last one left it.  All outputs are whole numbers.
"""
import numpy as np
import torch

import paper_1411_0127_gb300 as isg
from paper_1411_0127_gb300 import workloads

KINDS = ("minstd", "mt19937", "parisi_rapuano")
TEMPS = (0.5, 0.7, 0.9, 1.1, 1.5)
# 32-bit integer operations that one attempt cannot do without: the generator's
# recurrence and output, the comparison, and the bit-sliced logic's share
OPS = {"minstd": 11, "mt19937": 17, "parisi_rapuano": 16}


def listed():
    return [
        # the parity workload, a quench whose energy and spins are logged after
        # every sweep: launches and latency
        {"name": "quench_L32_minstd_each", "do": "quench", "L": 32, "rng": "minstd", "T": 1.1, "sweeps": 1},
        # a small lattice between two measurements (8 generator streams)
        {"name": "quench_L64_mt", "do": "quench", "L": 64, "rng": "mt19937", "T": 0.7, "sweeps": 32},
        # a ragged size with the third generator: rows that fill no word, a short last stream
        {"name": "quench_L150_pr", "do": "quench", "L": 150, "rng": "parisi_rapuano", "T": 0.9, "sweeps": 32},
        # the medium workload with both of its generators
        {"name": "quench_L256_minstd", "do": "quench", "L": 256, "rng": "minstd", "T": 0.7, "sweeps": 64},
        {"name": "quench_L256_mt", "do": "quench", "L": 256, "rng": "mt19937", "T": 0.7, "sweeps": 64},
        # the headline workload: the largest lattice in ordinary use, many sweeps a call
        {"name": "quench_L1024_mt", "do": "quench", "L": 1024, "rng": "mt19937", "T": 0.9, "sweeps": 64},
        # configurations that live on the host: spins in, one sweep, spins and
        # energy out, four lattices in flight
        {"name": "exchange_L1024_mt", "do": "exchange", "L": 1024, "rng": "mt19937", "T": 0.9, "sweeps": 1,
         "lattices": 4},
        # what is measured between runs: energies, overlap and hash of two replicas
        {"name": "measure_L512", "do": "measure", "L": 512, "rng": "minstd", "T": 0.9, "sweeps": 2},
        # the batched workload: disorder samples of mixed sizes, two replicas
        # each, 64 sweeps between measurements
        {"name": "batch_512x2_mt", "do": "batch", "samples": 512, "rng": "mt19937", "sweeps": 64},
        # multispin ensembles, 32 systems a word: one that memory bounds ...
        {"name": "amsc_L512_mt", "do": "amsc", "L": 512, "rng": "mt19937", "T": 0.9, "sweeps": 16},
        # ... and a small one with its spins read back
        {"name": "amsc_L64_minstd", "do": "amsc", "L": 64, "rng": "minstd", "T": 0.7, "sweeps": 64},
        # a burst of jobs of mixed size, generator and length, served to the end
        {"name": "serve_24_jobs", "do": "serve", "jobs": 24, "Lmax": 256, "sweeps_max": 512},
    ]


def _even(rng, lo, hi):
    """An even size, spread over the logarithm of [lo, hi]; half of the draws any even number, half a multiple of 16."""
    v = lo * (hi / lo) ** rng.random()
    step = 16 if rng.random() < 0.5 and lo >= 16 else 2
    return int(min(hi, max(lo, step * round(v / step))))


def _sweeps(rng, most):
    return int(max(1, min(most, round(most ** rng.random()))))


def draw(rng):
    do = rng.choice(["quench", "quench", "quench", "quench", "quench", "exchange", "measure", "batch", "amsc", "amsc",
                     "serve"])
    kind = rng.choice(KINDS)
    if do == "quench":
        L = _even(rng, 16, 1024)
        return {"do": do, "L": L, "rng": kind, "T": rng.choice(TEMPS),
                "sweeps": _sweeps(rng, min(256, 2 ** 36 // L ** 3))}
    if do == "exchange":
        return {"do": do, "L": _even(rng, 32, 1024), "rng": kind, "T": rng.choice(TEMPS), "sweeps": rng.randint(1, 4),
                "lattices": rng.randint(1, 4)}
    if do == "measure":
        return {"do": do, "L": _even(rng, 32, 1024), "rng": "minstd", "T": rng.choice(TEMPS), "sweeps": 2}
    if do == "batch":
        return {"do": do, "samples": int(round(8 * 64 ** rng.random())), "rng": kind, "sweeps": _sweeps(rng, 64)}
    if do == "amsc":
        L = _even(rng, 16, 512)
        return {"do": do, "L": L, "rng": kind, "T": rng.choice(TEMPS), "sweeps": _sweeps(rng, min(128, 2 ** 32 // L ** 3))}
    return {"do": do, "jobs": rng.randint(4, 32), "Lmax": 16 * rng.randint(4, 16), "sweeps_max": _sweeps(rng, 1024)}


def _pinned(n, dtype):
    return torch.empty(n, dtype=dtype, pin_memory=True).numpy()


def _seeds(seed):
    return 1000 + 64 * int(seed), 2000 + 64 * int(seed)


def _jobs(case, seed):
    """Jobs with the serving workload's distributions, cut at the case's sizes."""
    g = np.random.default_rng(seed)
    out = []
    for j in range(case["jobs"]):
        L = int(g.choice(np.arange(32, case["Lmax"] + 1, 16)))
        sweeps = int(10 ** g.uniform(0, np.log10(case["sweeps_max"]))) if case["sweeps_max"] > 1 else 1
        out.append((L, 50_000 + 100 * seed + j, 90_000 + 100 * seed + j, 1.0 / float(g.uniform(0.5, 1.5)),
                    KINDS[int(g.integers(0, 2))], max(1, sweeps)))
    return out


_installed = []


def prepare(case, seed):
    if not _installed:  # once per process: handles keep the allocator they were made with
        isg.use_torch_allocator()
        _installed.append(True)
    do = case["do"]
    sJ, sS = _seeds(seed)
    st = {"case": case}
    if do == "quench":
        st["sim"] = isg.Sim(case["L"], sJ, sS, 1.0 / case["T"], case["rng"])
        st["bits"] = _pinned((case["L"] ** 3 + 7) // 8, torch.uint8)
        st["E"] = _pinned(1, torch.int64)
    elif do == "exchange":
        nb = (case["L"] ** 3 + 7) // 8
        st["sims"] = [isg.Sim(case["L"], sJ, sS + m, 1.0 / case["T"], case["rng"]) for m in range(case["lattices"])]
        g = torch.Generator().manual_seed(int(seed))
        st["in"] = [_pinned(nb, torch.uint8) for _ in st["sims"]]
        # whole bytes of random spins (L even: L^3 is a multiple of 8, no bit is left over)
        block = torch.randint(0, 256, (min(nb, 1 << 22),), dtype=torch.uint8, generator=g).numpy()
        for m, b in enumerate(st["in"]):
            b[:] = np.resize(np.roll(block, 977 * m), nb)
        st["out"] = [_pinned(nb, torch.uint8) for _ in st["sims"]]
        st["E"] = [_pinned(1, torch.int64) for _ in st["sims"]]
        st["streams"] = [torch.cuda.Stream() for _ in st["sims"]]
    elif do == "measure":
        st["pair"] = [isg.Sim(case["L"], sJ, sS + m, 1.0 / case["T"], case["rng"]) for m in range(2)]
        for s in st["pair"]:
            s.sweep(case["sweeps"])
    elif do == "batch":
        ss = workloads.batch_samples(case["samples"], sampler_seed=7)
        st["batch"] = isg.Batch([s.L for s in ss], [s.seed_J + 1000 * int(seed) for s in ss],
                                [v + 2048 * int(seed) for s in ss for v in s.seed_spin], [1.0 / s.T for s in ss],
                                case["rng"])
    elif do == "amsc":
        J, S = workloads.amsc_seeds(case["L"])
        st["ens"] = isg.Amsc(case["L"], [v + 4096 * int(seed) for v in J], [v + 4096 * int(seed) for v in S], sS,
                             1.0 / case["T"], case["rng"])
    else:
        st["jobs"] = _jobs(case, int(seed))
    torch.cuda.synchronize()
    return st


def run(st):
    case = st["case"]
    do = case["do"]
    if do == "quench":
        st["sim"].exchange_async(None, st["bits"], case["sweeps"], st["E"])
        return [st["bits"], st["E"]]
    if do == "exchange":
        here = torch.cuda.current_stream()
        for sim, i, o, E, s in zip(st["sims"], st["in"], st["out"], st["E"], st["streams"]):
            s.wait_stream(here)
            sim.exchange_async(i, o, case["sweeps"], E, stream=s)
        for s in st["streams"]:
            here.wait_stream(s)
        return [st["out"], st["E"]]
    if do == "measure":
        a, b = st["pair"]
        return [a.energy(), b.energy(), a.overlap(b), np.uint64(a.hash()).view(np.int64),
                np.uint64(b.hash()).view(np.int64)]
    if do == "batch":
        st["batch"].run(case["sweeps"], 64)
        E, Q = st["batch"].measure()
        tracked, H = st["batch"].tracked()
        return [E, Q, tracked, H.view(np.int64)]
    if do == "amsc":
        st["ens"].sweep(case["sweeps"])
        out = [st["ens"].energies()]
        if case["L"] <= 64:
            out.append([st["ens"].spins(b) for b in range(isg.Amsc.SAMPLES)])
        return out
    srv = isg.Server(hbm_budget_bytes=150 * 10 ** 9, quantum_sweeps=64)
    ids = [srv.submit(*job) for job in st["jobs"]]
    srv.run()
    res = [srv.job(j) for j in ids]
    srv.close()
    return [np.array([[r["status"], r["E"]] for r in res], dtype=np.int64),
            np.array([r["H"] for r in res], dtype=np.uint64).view(np.int64)]


def work(case):
    """Bytes: the bit planes (spins and three couplings a site) read once, the spins written once, what crosses to and
    from the host; flops: the 32-bit integer operations of the attempts (see OPS)."""
    do = case["do"]
    if do in ("quench", "exchange"):
        n = case["L"] ** 3
        m = case.get("lattices", 1)
        planes = n / 8 * 5
        moved = n / 8 * (2 if do == "exchange" else 1)
        return {"bytes": m * (planes + moved), "flops": float(m * n * case["sweeps"] * OPS[case["rng"]])}
    if do == "measure":
        # two energies (4 bits a site), one overlap, two hashes (1 bit a site each)
        n = case["L"] ** 3
        return {"bytes": n / 8 * 12.0, "flops": 2.0 * n}
    if do == "batch":
        n = sum(2 * s.L ** 3 for s in workloads.batch_samples(case["samples"], sampler_seed=7))
        return {"bytes": n / 8 * 5, "flops": float(n * case["sweeps"] * OPS[case["rng"]])}
    if do == "amsc":
        n = case["L"] ** 3
        # one draw a site for the 32 systems, about 50 word operations for their updates
        return {"bytes": 4.0 * n * 5 * case["sweeps"], "flops": float(n * case["sweeps"] * (OPS[case["rng"]] + 50))}
    jobs = _jobs(case, 1)
    return {"bytes": sum(j[0] ** 3 for j in jobs) / 8 * 5.0,
            "flops": float(sum(j[0] ** 3 * j[5] * OPS[j[4]] for j in jobs))}


# ------------------------------------------------------------------ exact ---
_M64 = (1 << 64) - 1


def _sm64(seed, n):
    """Output n (an array) of the SplitMix64 generator whose state starts at seed."""
    with np.errstate(over="ignore"):
        z = np.uint64(seed & _M64) + (n.astype(np.uint64) + np.uint64(1)) * np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        return z ^ (z >> np.uint64(31))


def exact(case, seed):
    """The first pass on a new lattice in plain numpy, for quenches of at most 2^24 attempts with the two common
    generators: the model's definitions, site by site (int8 spins and couplings, 64-bit draws and sums)."""
    if case["do"] != "quench" or case["rng"] == "parisi_rapuano" or case["L"] ** 3 * case["sweeps"] > 1 << 24:
        return None
    L = case["L"]
    N, half, rows = L ** 3, L // 2, L * L
    sJ, sS = _seeds(seed)
    i = np.arange(N, dtype=np.uint64)

    def sign(v):
        return np.where(v >> np.uint64(63), -1, 1).astype(np.int8).reshape(L, L, L)      # [z, y, x]

    J = [sign(_sm64(sJ ^ 0x6A09E667F3BCC908, 3 * i + np.uint64(d))) for d in range(3)]   # towards +x, +y, +z
    s = sign(_sm64(sS ^ 0xBB67AE8584CAA73B, i))
    S0 = min(8192, max(1, N // 32768))
    R = -(-rows // S0)                                                                   # rows of one stream
    S = -(-rows // R)
    v = _sm64(sS ^ 0x3C6EF372FE94F82B, np.arange(S, dtype=np.uint64))
    if case["rng"] == "mt19937":
        gens = [np.random.RandomState(int(x) & 0xFFFFFFFF)._bit_generator for x in v]

        def draws(t, n):
            return gens[t].random_raw(n).astype(np.int64)
    else:
        M = (1 << 31) - 1
        states = [1 + int(x) % (M - 1) for x in v]
        most = R * half
        power = np.empty(most, dtype=np.uint64)                                          # 16807^(j+1) mod M
        power[0] = 16807
        k = 1
        while k < most:
            m = min(k, most - k)
            power[k:k + m] = power[:m] * power[k - 1] % np.uint64(M)
            k += m

        def draws(t, n):
            x = power[:n] * np.uint64(states[t]) % np.uint64(M)
            states[t] = int(x[-1])
            return 2 * x.astype(np.int64)
    thr = [int(np.floor(2.0 ** 32 * np.exp(-4.0 * k / case["T"]))) for k in (1, 2, 3)]
    z, y, x = np.indices((L, L, L))
    colour = (x + y + z) & 1
    axes = (2, 1, 0)
    for _ in range(case["sweeps"]):
        for c in (0, 1):
            d = np.concatenate([draws(t, (min(rows, (t + 1) * R) - t * R) * half) for t in range(S)])
            u = np.zeros((L, L, L), dtype=np.int8)                                       # unsatisfied bonds
            for a, Jd in zip(axes, J):
                u += Jd * s * np.roll(s, -1, a) < 0
                u += np.roll(Jd * s, 1, a) * s < 0
            m = colour == c
            uc, sc = u[m], s[m]                                                          # rows in order, ascending x
            flip = (uc >= 3) | ((uc == 2) & (d < thr[0])) | ((uc == 1) & (d < thr[1])) | ((uc == 0) & (d < thr[2]))
            s[m] = np.where(flip, -sc, sc)
    E = -sum(int((Jd.astype(np.int64) * s * np.roll(s, -1, a)).sum()) for a, Jd in zip(axes, J))
    return [np.packbits(s.reshape(-1) > 0, bitorder="little"), np.array([E], dtype=np.int64)]
