"""Performance cases of the parallel multicanonical library: the calls its users make.

Every case goes through the package's public classes (Muca, MucaBatch).  Kinds:

  iterate   weight iterations (sweeps, merged histogram, ln W recursion), either from the
            infinite-temperature start with ln W = 0 ("start") or with the weights of a
            run in progress ("late": the model's own entropy plus statistical noise)
  measure   thermalisation, production sweeps with (E, M) records, reweighting of the
            records to a grid of inverse temperatures
  batch     weight iterations of many lattices at once
  reweight  reweighting alone, of given production sums

Chains, histograms and records are integers fixed by the seed; ln W and the reweighted
observables are FP64.
"""
import math

import numpy as np
import torch

import paper_1212_3975_gb300 as muca

ISING_BETA0 = 0.4406867935097715   # ln(1 + sqrt 2) / 2
POTTS_BETA0 = 1.3424540464535260   # ln(1 + sqrt 8)


def listed():
    return [
        # a small lattice's first iterations: launches and latency (statistical studies run thousands)
        dict(name="start_ising_L8_p8", kind="iterate", model="ising", L=8, p=8, sweeps=200, rounds=3, weights="start"),
        # the plain workload from its start: every chain at infinite temperature, ln W = 0
        dict(name="start_ising_L64_p1024", kind="iterate", model="ising", L=64, p=1024, sweeps=25, rounds=4,
             weights="start"),
        # one later iteration of the plain workload (most of a run)
        dict(name="iterate_ising_L64_p1024", kind="iterate", model="ising", L=64, p=1024, sweeps=40, rounds=1,
             weights="late"),
        # the plain workload's measurement: thermalisation, records, FP64 reweighting
        dict(name="measure_ising_L64_p1024", kind="measure", model="ising", L=64, p=1024, therm=10, sweeps=40,
             betas=512, prec="fp64", weights="late"),
        # as many chains as fill the GPU
        dict(name="iterate_ising_L64_p14592", kind="iterate", model="ising", L=64, p=14592, sweeps=20, rounds=1,
             weights="late"),
        # a lattice side that is not a multiple of four, a ragged number of chains
        dict(name="iterate_ising_L90_p700", kind="iterate", model="ising", L=90, p=700, sweeps=10, rounds=1,
             weights="late"),
        # large lattices at fixed weights, records reweighted to many temperatures
        dict(name="measure_ising_L256_p8192", kind="measure", model="ising", L=256, p=8192, therm=0, sweeps=4,
             betas=4096, prec="fp32", weights="canonical"),
        # 8-state Potts: a later iteration with many chains
        dict(name="iterate_potts_L32_p4096", kind="iterate", model="potts", L=32, p=4096, sweeps=40, rounds=1,
             weights="late"),
        # 8-state Potts at fixed weights on a large lattice
        dict(name="measure_potts_L128_p4096", kind="measure", model="potts", L=128, p=4096, therm=0, sweeps=4,
             betas=4096, prec="fp32", weights="canonical"),
        # many lattices of uneven size and both models in one object
        dict(name="batch_mixed", kind="batch", ising="16,24,32,48,64,96,128", potts="16,24,32,48", p=256, sweeps=10,
             rounds=2),
        # reweighting alone: the plain workload's grid in FP64, a large lattice's in FP32
        dict(name="reweight_ising_L64_fp64", kind="reweight", model="ising", L=64, betas=512, prec="fp64",
             shape="flat"),
        dict(name="reweight_ising_L256_fp32", kind="reweight", model="ising", L=256, betas=4096, prec="fp32",
             shape="canonical"),
    ]


def _spread(rng, lo, hi):
    """Whole number between lo and hi, uniform in its logarithm."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["iterate", "iterate", "iterate", "measure", "measure", "batch", "reweight"])
    if kind == "batch":
        sides = rng.sample([16, 20, 24, 32, 36, 48, 64, 96, 128], rng.randint(3, 6))
        q8 = rng.sample([8, 12, 16, 24, 32, 40, 48], rng.randint(2, 4))
        return dict(kind=kind, ising=",".join(map(str, sorted(sides))), potts=",".join(map(str, sorted(q8))),
                    p=_spread(rng, 40, 256), sweeps=rng.randint(4, 10), rounds=rng.randint(1, 2))
    model = rng.choice(["ising", "ising", "potts"])
    if kind == "reweight":
        L = 2 * _spread(rng, 8, 128) if model == "ising" else _spread(rng, 12, 128)
        return dict(kind=kind, model=model, L=L, betas=_spread(rng, 33, 4096), prec=rng.choice(["fp64", "fp32"]),
                    shape=rng.choice(["flat", "canonical"]))
    # half of the sides are whole 32-site words, as in the configurations; the others are any
    if model == "ising":
        L = rng.choice([32, 64, 96, 128, 160, 256]) if rng.random() < 0.5 else 2 * _spread(rng, 4, 64)
    else:
        L = rng.choice([32, 64, 96, 128]) if rng.random() < 0.5 else _spread(rng, 5, 128)
    V = L * L
    most = min(16384, 2 ** 29 // V)
    p = _spread(rng, 8, most)
    sweeps = max(2, min(200, 2 ** 16 // V, 2 ** 29 // (V * p)))
    if kind == "iterate":
        return dict(kind=kind, model=model, L=L, p=p, sweeps=sweeps, rounds=1, weights=rng.choice(["late", "start"]))
    return dict(kind=kind, model=model, L=L, p=p, therm=rng.choice([0, 2]), sweeps=sweeps,
                betas=_spread(rng, 33, 1024), prec=rng.choice(["fp64", "fp32"]),
                weights=rng.choice(["late", "canonical"]))


# -- weights and production sums --------------------------------------------------------


def _bins(model, L):
    V = L * L
    b = np.arange(V + 1 if model == "ising" else 2 * V + 1)
    E = (4.0 * b if model == "ising" else 1.0 * b) - 2.0 * V
    acc = np.ones(len(b), dtype=bool)
    if model == "ising":
        acc[[1, -2]] = False
    else:
        acc[[1, 2, 3, 5]] = False
    return E, acc


def _ising_energy(beta):
    """Energy per site of the infinite square lattice (Onsager), by the AGM."""
    beta = np.asarray(beta, dtype=np.float64)
    k = 2 * np.sinh(2 * beta) / np.cosh(2 * beta) ** 2
    a, b = np.ones_like(k), np.sqrt(np.maximum(1 - k * k, 1e-12))
    for _ in range(12):
        a, b = 0.5 * (a + b), np.sqrt(a * b)
    K1 = np.pi / (2 * a)
    th = np.tanh(2 * beta)
    return -(1 / th) * (1 + 2 / np.pi * (2 * th * th - 1) * K1)


def _inverse_temperature(model, e):
    """Microcanonical inverse temperature of energy per site e."""
    if model == "ising":
        beta = np.linspace(1e-3, 1.6, 4001)
        en = np.concatenate([_ising_energy(beta)[::-1], [0.0], -_ising_energy(beta)])
        return np.interp(e, en, np.concatenate([beta[::-1], [0.0], -beta]))
    # 8-state Potts: high-temperature values, the coexistence interval at beta_0, low energies
    en = [-2.0, -1.9, -1.8, -1.5967, -1.1104, -0.95, -0.75, -0.57, -0.40, -0.25, -0.12, 0.0]
    be = [2.2, 1.65, 1.48, POTTS_BETA0, POTTS_BETA0, 1.31, 1.20, 0.98, 0.55, 0.0, -0.8, -3.0]
    return np.interp(e, en, be)


def _lnw(model, L, weights, rng):
    E, acc = _bins(model, L)
    if weights == "canonical":
        lnw = -(ISING_BETA0 if model == "ising" else POTTS_BETA0) * E
    else:
        beta = _inverse_temperature(model, E / (L * L))
        steps = 0.5 * (beta[1:] + beta[:-1]) * np.diff(E)
        lnw = -np.concatenate([[0.0], np.cumsum(steps)]) + rng.normal(0.0, 0.01, len(E))
    return np.where(acc, lnw - lnw[acc].max(), 0.0)


def _sums(model, L, shape, rng):
    """Production sums (records, sum |M|, sum M^2 per bin) and the weights they belong to."""
    E, acc = _bins(model, L)
    V = L * L
    beta = _inverse_temperature(model, E / V)
    S = np.concatenate([[0.0], np.cumsum(0.5 * (beta[1:] + beta[:-1]) * np.diff(E))])
    lnw = _lnw(model, L, "canonical", rng) if shape == "canonical" else np.where(acc, -S - (-S)[acc].max(), 0.0)
    lnp = np.where(acc, S + lnw, -np.inf)
    prob = np.exp(lnp - lnp.max())
    n = rng.multinomial(8_000_000, prob / prob.sum()).astype(np.int64)
    top = V if model == "ising" else 7 * V
    mean = np.clip(-0.6 * E / V if model == "ising" else -E / V - 0.5, 0.02, 0.98) * top
    s1 = np.rint(n * mean).astype(np.int64)
    s2 = np.rint(n * (mean ** 2 + (0.02 * top) ** 2)).astype(np.int64)
    return n, s1, s2, lnw


def _grid(model, count):
    lo, hi = (0.3, 0.6) if model == "ising" else (1.2, 1.4)
    return np.linspace(lo, hi, count)


# -- prepare / run ------------------------------------------------------------------------


def _model(name):
    return (muca.MUCA_ISING, 2) if name == "ising" else (muca.MUCA_POTTS, 8)


def _stream():
    return torch.cuda.current_stream().cuda_stream


def prepare(case, seed):
    rng = np.random.default_rng(seed)
    st = dict(case=case, seed=int(seed) % (1 << 31) + 1)
    kind = case["kind"]
    if kind == "batch":
        jobs = [(muca.MUCA_ISING, int(L), 2, case["p"], st["seed"]) for L in case["ising"].split(",")]
        jobs += [(muca.MUCA_POTTS, int(L), 8, case["p"], st["seed"]) for L in case["potts"].split(",")]
        st["batch"] = b = muca.MucaBatch(jobs, stream=_stream())
        for j, (model, L, _, _, _) in enumerate(jobs):
            b.job(j).set_lnw(_lnw("ising" if model == muca.MUCA_ISING else "potts", L, "late", rng))
        return st
    model, L = case["model"], case["L"]
    m, q = _model(model)
    g = st["ctx"] = muca.Muca(m, L, q, case.get("p", 1), st["seed"], stream=_stream())
    if kind == "reweight":
        n, s1, s2, lnw = _sums(model, L, case["shape"], rng)
        g.set_lnw(lnw)
        g.set_samples(n, s1, s2)
    elif case["weights"] != "start":
        g.set_lnw(_lnw(model, L, case["weights"], rng))
        # chains in the middle of a run: spread over the energies by earlier sweeps
        g.thermalize(max(4, min(400, 2 ** 22 // (L * L), 2 ** 33 // (L * L * case["p"]))))
    if kind == "iterate":
        st["H"] = torch.zeros(g.n_bins, dtype=torch.int64, device="cuda")
    else:
        st["betas"] = torch.tensor(_grid(model, case["betas"]), dtype=torch.float64, device="cuda")
        st["obs"] = torch.zeros((4, case["betas"]), dtype=torch.float64, device="cuda")
    if kind == "measure":
        st["E"], st["M"] = (torch.zeros((case["sweeps"], case["p"]), dtype=torch.int32, device="cuda")
                            for _ in range(2))
    return st


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "batch":
        b = st["batch"]
        b.iterate(case["rounds"], case["sweeps"])
        out = {}
        for j in range(len(b)):
            out["H%d" % j] = b.job(j).get_histogram().view(np.int64)
            out["lnw%d" % j] = b.job(j).get_lnw()
        return out
    g = st["ctx"]
    if kind == "iterate":
        if case["weights"] == "start":
            g.reset(st["seed"])
        for _ in range(case["rounds"]):
            g.iterate(case["sweeps"], H_out=st["H"])
            stats = g.update_weights()
        E, M = g.get_energies()
        return dict(H=st["H"], lnw=g.get_lnw(), E=E, M=M, sampled=int(stats["n_sampled"]), flat=int(stats["flat"]))
    if kind == "measure":
        if case["therm"]:
            g.thermalize(case["therm"])
        g.produce(case["sweeps"], E_out=st["E"], M_out=st["M"])
        g.reweight(st["betas"], case["prec"], out=st["obs"])
        return dict(E=st["E"], M=st["M"], e=st["obs"][0], C=st["obs"][1], absm=st["obs"][2], chi=st["obs"][3])
    g.reweight(st["betas"], case["prec"], out=st["obs"])
    return dict(e=st["obs"][0], C=st["obs"][1], absm=st["obs"][2], chi=st["obs"][3])


# -- what a pass cannot do without ----------------------------------------------------------


def _sweep_work(model, L, p, sweeps):
    """Integer operations and lattice bytes of `sweeps` sweeps: per attempt its share of
    the random block (10 rounds of 4 products and sums for 4 / 2 attempts), the
    neighbours and the test; every lattice read and written once per launch."""
    V = L * L
    ops = (10 + 10 if model == "ising" else 20 + 15) * V * p * sweeps
    return 2.0 * p * (V / 8 if model == "ising" else V), float(ops)


def work(case):
    kind = case["kind"]
    if kind == "batch":
        jobs = [("ising", int(L)) for L in case["ising"].split(",")] + [("potts", int(L)) for L in
                                                                        case["potts"].split(",")]
        by = fl = 0.0
        for model, L in jobs:
            b, f = _sweep_work(model, L, case["p"], case["sweeps"])
            nb = len(_bins(model, L)[0])
            by += case["rounds"] * (b + 24.0 * nb)
            fl += case["rounds"] * (f + 20.0 * nb)
        return dict(bytes=by, flops=fl)
    nb = len(_bins(case["model"], case["L"])[0])
    if kind == "iterate":
        b, f = _sweep_work(case["model"], case["L"], case["p"], case["sweeps"])
        # histogram written, ln W and its accumulator updated
        return dict(bytes=case["rounds"] * (b + 40.0 * nb), flops=case["rounds"] * (f + 20.0 * nb))
    # reweighting: the sums and weights in, one exponential and six columns per (beta, bin
    # that carries weight); bins far from a beta's peak need none
    peak = min(nb, int(16 * math.sqrt(nb)))
    by, fl = 32.0 * nb + 40.0 * case["betas"], 14.0 * case["betas"] * peak
    if kind == "measure":
        b, f = _sweep_work(case["model"], case["L"], case["p"], case["sweeps"] + case["therm"])
        by, fl = by + b + 8.0 * case["p"] * case["sweeps"], fl + f
    return dict(bytes=by, flops=fl)


def exact(case, seed):
    """Reweighting in plain FP64 numpy (terms centred on their own means); the chains'
    outputs are integers, and what follows from them has no closed form."""
    if case["kind"] != "reweight":
        return None
    model, L, V = case["model"], case["L"], case["L"] ** 2
    n, s1, s2, lnw = _sums(model, L, case["shape"], np.random.default_rng(seed))
    E, _ = _bins(model, L)
    k = n > 0
    E, n, s1, s2, lnw = E[k], n[k].astype(np.float64), s1[k], s2[k], lnw[k]
    top = V if model == "ising" else 7 * V
    m1 = s1 / n / top
    # within-bin variance from the exact integers
    var = np.array([float(int(a) * int(c) - int(b) ** 2) for a, b, c in zip(n, s1, s2)]) / (n * top) ** 2
    G = np.log(n) - lnw
    out = {x: [] for x in ("e", "C", "absm", "chi")}
    for beta in _grid(model, case["betas"]):
        a = G - beta * E
        w = np.exp(a - a.max())
        w /= w.sum()
        em, mm = float(w @ E), float(w @ m1)
        out["e"].append(em / V)
        out["C"].append(beta ** 2 * float(w @ (E - em) ** 2) / V)
        out["absm"].append(mm)
        out["chi"].append(beta * V * float(w @ (var + (m1 - mm) ** 2)))
    return {x: np.array(v) for x, v in out.items()}
