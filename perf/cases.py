"""Workloads that the framework is measured on.

Each case is one call sequence of a user's program, from the host arrays of a
disorder instance to the numbers that the program keeps: a population is
created, annealed and read, or a gradient is taken, or a batch of instances is
annealed, or one resampling step runs on caller-owned device buffers.  All of
it goes through the package's public functions.

A case is a plain dict:

  what       anneal | overlap | beta_f | batch | resample
  D, L, R    lattice dimension and size, replicas (batch: per instance)
  couplings  pm (+-J) | gauss | pm_field (+-J with a uniform random field)
  T, n       temperatures of the full schedule, and how many of them are run
  beta       last inverse temperature of the full schedule
  sweeps     Metropolis sweeps per temperature

and, where they apply, storage (packed | i8), spins (configurations are read
back at the end), stepwise (observables are read after every temperature),
own_memory (the device memory is a torch tensor that the program keeps from one
instance to the next), grad (population counts and their backward pass), icm
(cluster moves), nearest (nearest-integer resampling with the dynamic population
of Eq. 6), instances (batch).
"""
import math

import numpy as np
import torch

import paper_1710_09025_gb300 as P
from paper_1710_09025_gb300 import schedules as S
from paper_1710_09025_gb300 import workloads as W
from paper_1710_09025_gb300.autograd import beta_f

BATCH_SIZES = (4, 6, 8, 10)


def _case(name, what, **kw):
    return dict({"name": name, "what": what, "sweeps": 10}, **kw)


def listed():
    return [
        # one resampling step on the caller's own device buffers, for hosts that
        # own all device memory: the smallest call, all launch latency
        _case("resample_static_r4096", "resample", L=8, R=4096),
        # the smallest population of the benchmark list (int8 storage), annealed
        # once per disorder instance in memory that is kept between instances
        _case("pm3d_l4_r1000_i8", "anneal", D=3, L=4, R=1000, couplings="pm", T=101, n=101, beta=5.0,
              storage="i8", spins=True, own_memory=True),
        # two independent populations of one instance and their overlap
        # histogram: the order parameter of a spin-glass study
        _case("pm3d_l8_r1e5_overlap", "overlap", D=3, L=8, R=100_000, couplings="pm", T=201, n=201, beta=5.0),
        # the largest workload of the benchmark list, its high-temperature stage
        # (the steps in which most random bits are drawn)
        _case("pm3d_l16_r1e6_hot", "anneal", D=3, L=16, R=1_000_000, couplings="pm", T=301, n=25, beta=5.0),
        # the same lattice with a tenth of the replicas over the whole schedule:
        # the low temperatures weigh as they do in a complete run
        _case("pm3d_l16_r1e5", "anneal", D=3, L=16, R=100_000, couplings="pm", T=301, n=301, beta=5.0),
        # a ragged population that is watched while it anneals: the observables
        # are read back after every temperature
        _case("pm3d_l12_r77777_watched", "anneal", D=3, L=12, R=77_777, couplings="pm", T=201, n=101, beta=5.0,
              stepwise=True),
        # one Gaussian instance of the disorder batch at its largest size
        _case("gauss3d_l10_r2e4", "anneal", D=3, L=10, R=20_000, couplings="gauss", T=201, n=201, beta=5.0),
        # the differentiation workload: free energy forward, gradient with
        # respect to every coupling backward, through autograd
        _case("gauss3d_l6_r5e4_grad", "beta_f", D=3, L=6, R=50_000, couplings="gauss", T=101, n=101, beta=3.0),
        # the small differentiation workload with a field on every site
        _case("pmfield2d_l4_r5e4_grad", "beta_f", D=2, L=4, R=50_000, couplings="pm_field", T=101, n=101, beta=3.0),
        # disorder average: many instances of mixed size and coupling kind in one
        # batch
        _case("batch64_mixed_r2e4", "batch", D=3, R=20_000, instances=64, T=201, n=31, beta=5.0),
        # two-dimensional lattice with isoenergetic cluster moves
        _case("pm2d_l32_r2e4_icm", "anneal", D=2, L=32, R=20_000, couplings="pm", T=101, n=101, beta=3.0, icm=True),
        # population that fluctuates around a shrinking target, configurations
        # kept at the last temperature
        _case("pm3d_l6_r40001_nearest", "anneal", D=3, L=6, R=40_001, couplings="pm", T=101, n=101, beta=5.0,
              nearest=True, spins=True),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    what = rng.choice(["anneal", "anneal", "anneal", "overlap", "beta_f", "batch", "resample"])
    if what == "resample":
        return {"what": what, "L": rng.choice([4, 6, 8, 10, 12]), "R": _log_int(rng, 100, P.PA_STATIC_MAX_R), "sweeps": 10}
    T = rng.choice([51, 101, 201, 301])
    case = {"what": what, "sweeps": rng.choice([1, 5, 10, 10]), "T": T, "beta": rng.choice([3.0, 5.0])}
    if what == "batch":
        case.update(D=3, instances=_log_int(rng, 4, 96), R=_log_int(rng, 500, 20_000), n=_log_int(rng, 8, 32))
        return case
    if what == "overlap":
        case.update(D=3, L=rng.choice([4, 6, 8, 10]), couplings="pm")
    elif what == "beta_f":
        case.update(rng.choice([dict(D=2, L=4), dict(D=2, L=8), dict(D=3, L=4), dict(D=3, L=6), dict(D=3, L=8)]))
        case.update(couplings=rng.choice(["gauss", "pm_field"]))
    else:
        case.update(rng.choice([dict(D=3, L=4), dict(D=3, L=6), dict(D=3, L=8), dict(D=3, L=10), dict(D=3, L=12),
                                dict(D=3, L=16), dict(D=2, L=8), dict(D=2, L=16), dict(D=2, L=32)]))
        case.update(couplings=rng.choice(["pm", "pm", "gauss"]))
        if case["couplings"] == "gauss" and case["L"] == 16 and case["D"] == 3:
            case["L"] = 12  # the largest lattice with real couplings
        extra = rng.choice(["", "", "i8", "grad", "icm", "nearest", "stepwise"])
        if extra == "i8":
            case["storage"] = "i8"
        elif extra:
            case[extra] = True
    # replicas over the range of the benchmark list, then as many of the
    # schedule's temperatures as keep the run below the listed ones
    real = case["couplings"] != "pm"
    N = case["L"] ** case["D"]
    case["R"] = _log_int(rng, 200, min(1e6, (5e7 if real else 1e9) / N))
    budget = 1e10 if real else 2e11
    if case.get("icm"):
        budget /= 10.0
    most = int(budget / (N * case["R"] * case["sweeps"]))
    case["n"] = max(2, min(T, most))
    return case


def _instance(D, L, couplings, seed):
    """(kind, J, h) of one disorder instance."""
    if couplings == "gauss":
        return P.PA_REAL, W.couplings_gauss(D, L, seed), None
    J = W.couplings_pm(D, L, seed)
    if couplings == "pm_field":
        return P.PA_REAL, J, W.field_uniform(L ** D, seed + 1)
    return P.PA_PM1, J, None


def _energies(case, seed):
    """Energies of a +-J population at one temperature: spread as in a run,
    congruent modulo 4 as they are for every population."""
    N = case["L"] ** 3
    g = torch.Generator(device="cuda").manual_seed(seed)
    z = torch.randn(case["R"], generator=g, device="cuda", dtype=torch.float64)
    e = (-1.2 * N + math.sqrt(3.0 * N) * z) / 4.0
    return (4 * torch.clamp(torch.round(e), -3 * N // 4, 3 * N // 4)).to(torch.int32)


RESAMPLE_BETAS = (0.80, 0.85)  # one step of a schedule near the middle of its range


def prepare(case, seed):
    st = {"case": case, "seed": seed, "stream": torch.cuda.Stream()}
    if case["what"] == "resample":
        st["E"] = _energies(case, seed)
        st["parent"] = torch.empty(case["R"], dtype=torch.int32, device="cuda")
        st["lnQ"] = torch.empty(1, dtype=torch.float64, device="cuda")
        return st
    st["betas"] = W.schedule_lb(case["T"], case["beta"])[: case["n"]]
    if case["what"] == "batch":
        st["instances"] = []
        for i in range(case["instances"]):
            L = BATCH_SIZES[(i // 2) % len(BATCH_SIZES)]
            kind, J, h = _instance(case["D"], L, "gauss" if i % 2 else "pm", seed * 1000 + i)
            st["instances"].append(dict(L=L, kind=kind, J=J, h=h, R=case["R"], rng_instance=i))
        return st
    kind, J, h = _instance(case["D"], case["L"], case["couplings"], seed)
    st.update(kind=kind, J=J, h=h, opts={})
    if case["what"] == "beta_f":
        st["J"] = torch.from_numpy(J).requires_grad_()
        st["h"] = None if h is None else torch.from_numpy(h).requires_grad_()
        st["gbar"] = torch.from_numpy(np.random.default_rng(seed).standard_normal(case["n"]))
        return st
    if case.get("storage"):
        st["opts"]["layout"] = {"packed": P.PA_LAYOUT_PACKED, "i8": P.PA_LAYOUT_I8}[case["storage"]]
    if case.get("grad"):
        st["opts"]["accumulate_grad"] = 1
        st["gbar"] = np.random.default_rng(seed).standard_normal(case["n"])
    if case.get("icm"):
        st["opts"]["icm"] = 1
    if case.get("nearest"):
        pops = np.maximum(1, np.rint(S.dps_population(st["betas"], case["R"], case["beta"]))).astype(np.int32)
        st["rows"] = case["R"] + 64 + 8 * math.ceil(math.sqrt(case["R"]))
        st["opts"].update(populations=pops, resampling=P.PA_RESAMPLE_NEAREST, capacity=st["rows"])
    if case.get("own_memory"):
        size = P.pa_workspace_size(case["D"], case["L"], kind, case["R"], case["n"], P.pa_options_default(**st["opts"]))
        st["memory"] = torch.empty(size + 256, dtype=torch.uint8, device="cuda")
    return st


def _create(st, **more):
    c = st["case"]
    a = (c["D"], c["L"], st["kind"], st["J"], st["h"], c["R"], st["betas"], c["sweeps"], st["seed"])
    opts = P.pa_options_default(**dict(st["opts"], **more))
    if "memory" not in st:
        return P.pa_create(*a, opts)
    at = (st["memory"].data_ptr() + 255) // 256 * 256
    return P.pa_create_ws(*a, at, st["memory"].data_ptr() + st["memory"].numel() - at, opts)


def _record(a, rows):
    """A population's array as a program files it: `rows` entries, those past
    the population 0 (it fluctuates under nearest-integer resampling)."""
    if rows is None:
        return a
    out = np.zeros((rows,) + a.shape[1:], a.dtype)
    out[: len(a)] = a
    return out


def _anneal(st):
    c = st["case"]
    rows = st.get("rows")
    with torch.cuda.stream(st["stream"]):
        ctx = _create(st)
    try:
        out = {}
        if c.get("stepwise"):
            seen = []
            while P.pa_anneal_step(ctx):
                seen.append(P.pa_observables(ctx, len(seen)))
            for key in ("E_mean", "E2_mean", "C", "lnQ", "S_f", "rho_s"):
                out[key] = np.array([o[key] for o in seen])
        else:
            P.pa_anneal(ctx)
            last = P.pa_observables(ctx, c["n"] - 1)
            out["last"] = np.array([last[key] for key in ("E_mean", "E2_mean", "C", "lnQ", "S_f", "rho_s")])
        out["betaF"] = P.pa_free_energy(ctx)
        out["energies"] = _record(P.pa_get_energies(ctx, st["kind"]), rows)
        out["family"] = _record(P.pa_get_family(ctx), rows)
        if c.get("spins"):
            out["spins"] = _record(P.pa_get_spins(ctx), rows)
        if c.get("grad"):
            out["dJ"], out["dh"] = P.pa_grad(ctx, st["gbar"])
        return out
    finally:
        P.pa_destroy(ctx)


def _overlap(st):
    ctx = []
    try:
        with torch.cuda.stream(st["stream"]):
            for tag in (0, 1):
                ctx.append(_create(st, rng_tag=tag))
        for c in ctx:
            P.pa_anneal(c)
        hist = P.pa_overlap(*ctx)
        return {"hist": hist, "betaF": [P.pa_free_energy(c) for c in ctx],
                "energies": [P.pa_get_energies(c, st["kind"]) for c in ctx]}
    finally:
        for c in ctx:
            P.pa_destroy(c)


def _beta_f(st):
    c = st["case"]
    J, h = st["J"], st["h"]
    J.grad = None
    if h is not None:
        h.grad = None
    bF = beta_f(J, h, c["D"], c["L"], c["R"], st["betas"], c["sweeps"], st["seed"])
    bF.backward(st["gbar"])
    out = {"betaF": bF, "dJ": J.grad}
    if h is not None:
        out["dh"] = h.grad
    return out


def _batch(st):
    c = st["case"]
    with torch.cuda.stream(st["stream"]):
        b = P.pa_batch_create(c["D"], st["instances"], st["betas"], c["sweeps"], st["seed"])
    try:
        P.pa_batch_run(b)
        bF, energies = [], []
        for i, inst in enumerate(st["instances"]):
            ctx = P.pa_batch_instance(b, i)
            bF.append(P.pa_free_energy(ctx))
            energies.append(P.pa_get_energies(ctx, inst["kind"]).reshape(c["R"], -1)[:, 0])
        return {"betaF": np.stack(bF), "energies": np.stack(energies)}
    finally:
        P.pa_batch_destroy(b)


def run(st):
    what = st["case"]["what"]
    if what == "resample":
        P.pa_resample_static(st["E"].data_ptr(), st["case"]["R"], *RESAMPLE_BETAS, 7, st["seed"], 0, 0,
                             st["parent"].data_ptr(), st["lnQ"].data_ptr())
        return {"parent": st["parent"], "lnQ": st["lnQ"]}
    return {"anneal": _anneal, "overlap": _overlap, "beta_f": _beta_f, "batch": _batch}[what](st)


def _anneal_work(D, L, couplings, R, n, sweeps):
    """One temperature reads and writes every replica once (a bit per +-J spin
    however it is stored, a byte per spin with real couplings) with its energy,
    parent and family; an attempted flip sums 2 D neighbours."""
    N = L ** D
    per_replica = N / 8 if couplings == "pm" else N
    record = 4 if couplings == "pm" else 16
    return {"bytes": float(n) * R * (2 * per_replica + 2 * record + 4 + 8) + 4.0 * D * N,
            "flops": float(n) * R * N * sweeps * 2 * D}


def work(case):
    if case["what"] == "resample":
        return {"bytes": 8.0 * case["R"] + 8.0, "flops": 2.0 * case["R"]}
    if case["what"] == "batch":
        parts = [_anneal_work(case["D"], BATCH_SIZES[(i // 2) % len(BATCH_SIZES)], "gauss" if i % 2 else "pm", case["R"],
                              case["n"], case["sweeps"]) for i in range(case["instances"])]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    w = _anneal_work(case["D"], case["L"], case["couplings"], case["R"], case["n"], case["sweeps"])
    return {k: v * (2 if case["what"] == "overlap" else 1) for k, v in w.items()}


def exact(case, seed):
    """ln Q = ln of the mean resampling weight, in 64 bits.  The floating
    outputs of the other cases are estimates from the run's own random numbers:
    no other program has values for them."""
    if case["what"] != "resample":
        return None
    x = -(RESAMPLE_BETAS[1] - RESAMPLE_BETAS[0]) * _energies(case, seed).to(torch.float64)
    return {"parent": None, "lnQ": (torch.logsumexp(x, 0) - math.log(case["R"])).reshape(1)}
