"""The performance cases: what users of this library have it do, through the
package's public entry points, from the smallest calls to the largest.

A case is a dict of plain values; `kind` says which call it stands for:

  rm        one Robbins-Monro iteration of a batch of window-restricted chains
            (Batch.rm_step), the call every study spends its time in
  rm_save   the same, then a checkpoint of the whole chain state (save_state)
  rm_run    several iterations as graph replays on device buffers (rm_run)
  exchange  one iteration, then a replica-exchange round (Sec. 2.5)
  muca      multicanonical sweeps with their energy history (Sec. 2.6)
  or_pass   one overrelaxation pass from given links (the layer that makes up
            four of the five passes of a composite sweep)
  load      stored configurations into a batch, their energies, and back
  recon     ln rho, action observables and the C_V peak from the slopes
  reweight  multicanonical samples reweighted to couplings, the C_V peak
  mlp_fit   the warm start: two trainings (held-out error, final), a prediction
  mlp_grad  loss and gradient of the warm-start network
"""
import math

import numpy as np
import torch

from paper_1509_08391_gb300 import llr, warmstart, workloads

# floating-point operations of one link update (six staple angles, their sines
# and cosines, the sums, the new angle), of one plaquette of the energy, and of
# one sample or centre at one coupling (exp and three sums)
FLOPS_OR, FLOPS_HB, FLOPS_PLAQUETTE, FLOPS_MOMENT = 60, 220, 35, 25
N_PARAMS = 8641


def _sweep_flops(n_or):
    """Of one composite sweep, per link."""
    return FLOPS_HB + n_or * FLOPS_OR + 1.5 * FLOPS_PLAQUETTE


LARGEST = 2048 * 4 * 20 ** 4 * 5 * _sweep_flops(4)   # the largest listed case


def listed():
    return [
        # the smallest workload: L = 4, 8 intervals, 50 + 100 sweeps a step;
        # every launch, barrier and dependent load counts
        _rm("rm_l4_8int", 4, 8, 1, 0.55, 0.70, 4.0, 50, 100),
        # the small overlapping-window study: short steps with an exchange round
        {"name": "exchange_l4_12", "kind": "exchange", "n_int": 6, "replicas": 2, "n_therm": 5,
         "n_meas": 20},
        # the small-volume batch (L = 8, 32 intervals x 4 replicas), checkpointed
        dict(_rm("rm_l8_128_save", 8, 32, 4, 0.58, 0.68, 8.0, 50, 100), kind="rm_save"),
        # lattices of three sizes in one launch, graph replays
        {"name": "run_uneven_192", "kind": "rm_run", "n_int": 64, "Ls": "8,12,16", "n_therm": 2,
         "n_meas": 8, "n_steps": 2},
        # the paper's volume study at L = 14 (half rows of odd length, 512
        # narrow contiguous intervals)
        _rm("rm_l14_512", 14, 512, 1, 0.59, 0.687777,
            6.0 * 14 ** 4 * (0.687777 - 0.59) / 512, 2, 8),
        # the benchmark's batch: L = 20, 256 intervals x 8 replicas, 5.2 GB of
        # links, one short step (1 + 4 sweeps)
        _rm("rm_l20_2048", 20, 256, 8, 0.62, 0.67, 12.0, 1, 4),
        # the multicanonical run: 512 chains, 64-interval table
        {"name": "muca_l8_512", "kind": "muca", "L": 8, "chains": 512, "n_int": 64,
         "sweeps": 20},
        # one overrelaxation pass of a few L = 16 lattices
        {"name": "or_pass_l16_8", "kind": "or_pass", "L": 16, "n": 8},
        # stored L = 20 configurations read back and measured
        {"name": "load_l20_8", "kind": "load", "L": 20, "n": 8},
        # the analysis of one finished study: 512 slopes
        {"name": "recon_512", "kind": "recon", "n": 512, "n_beta": 401, "n_grid": 1601},
        # the analysis of a multicanonical run: 512 chains x 1000 samples
        {"name": "reweight_512k", "kind": "reweight", "samples": 512000, "n_int": 64,
         "n_beta": 101, "n_grid": 201},
        # the warm start: 24 intervals at five volumes
        {"name": "mlp_fit_120", "kind": "mlp_fit", "n": 24, "epochs": 1000, "n_pred": 256},
    ]


def _rm(name, L, n_int, replicas, e_lo, e_hi, dE, n_therm, n_meas, n_or=4, block=1, fast=True):
    return {"name": name, "kind": "rm", "L": L, "n_int": n_int, "replicas": replicas,
            "e_lo": e_lo, "e_hi": e_hi, "dE": dE, "n_therm": n_therm, "n_meas": n_meas,
            "n_or": n_or, "block": block, "fast": fast}


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["rm"] * 6 + ["rm_save", "rm_run", "exchange", "muca", "muca", "or_pass",
                                    "load", "recon", "reweight", "mlp_fit", "mlp_grad"])
    if kind in ("rm", "rm_save"):
        L = rng.choice([4, 6, 8, 10, 12, 14, 16, 18, 20, 24])
        n_or = rng.choice([4, 4, 4, 4, 1, 2, 8])
        sweeps = _log_int(rng, 3, 60)
        fast = rng.random() > 0.1
        # bounded by the largest listed case, and by one lattice's serial work
        sweeps = max(2, min(sweeps, int(6e7 // (4 * L ** 4 * (n_or + 1)))))
        one = 4 * L ** 4 * sweeps * _sweep_flops(n_or)
        most = max(1, min(2048, int((0.9 if fast else 0.4) * LARGEST // one)))
        if kind == "rm_save":
            most = max(1, min(most, int(4e6 // (4 * L ** 4))))
        n_lat = _log_int(rng, 1, most)
        replicas = rng.choice([1, 1, 2, 4])
        n_int = max(1, n_lat // replicas)
        n_therm = rng.randrange(0, sweeps)
        c = _rm("", L, n_int, replicas, 0.58, 0.68, max(4.0, 8.0 * (L / 8) ** 2), n_therm,
                sweeps - n_therm, n_or, rng.choice([1, 1, 1, 1, 4]), fast)
        c["kind"] = kind
    elif kind == "rm_run":
        c = {"kind": kind, "n_int": _log_int(rng, 2, 96),
             "Ls": rng.choice(["8,12,16", "8,10,12,14,16", "4,8", "6,10,14", "8,20"]),
             "n_therm": rng.randrange(0, 4), "n_meas": rng.randrange(1, 9),
             "n_steps": rng.randrange(1, 4)}
    elif kind == "exchange":
        c = {"kind": kind, "n_int": rng.randrange(2, 10), "replicas": rng.choice([1, 2, 4, 8]),
             "n_therm": rng.randrange(0, 10), "n_meas": rng.randrange(5, 40)}
    elif kind == "muca":
        L = rng.choice([4, 6, 8, 10, 12])
        c = {"kind": kind, "L": L, "chains": _log_int(rng, 4, 512 if L <= 8 else 128),
             "n_int": rng.choice([16, 64, 128]),
             "sweeps": _log_int(rng, 2, max(4, min(100, 400000 // L ** 4)))}
    elif kind in ("or_pass", "load"):
        L = rng.choice([4, 6, 8, 10, 12, 14, 16, 18, 20, 22, 24])
        c = {"kind": kind, "L": L, "n": rng.randrange(1, 21 if L <= 16 else 9)}
    elif kind == "recon":
        c = {"kind": kind, "n": _log_int(rng, 24, 4096), "n_beta": _log_int(rng, 1, 1000),
             "n_grid": _log_int(rng, 101, 2001)}
    elif kind == "reweight":
        c = {"kind": kind, "samples": _log_int(rng, 3000, 700000),
             "n_int": rng.choice([16, 64, 128, 512]), "n_beta": _log_int(rng, 1, 200),
             "n_grid": rng.choice([101, 161, 201])}
    elif kind == "mlp_fit":
        c = {"kind": kind, "n": rng.randrange(6, 33), "epochs": _log_int(rng, 200, 2000),
             "n_pred": _log_int(rng, 8, 2048)}
    else:
        c = {"kind": kind, "n": _log_int(rng, 16, 1024)}
    return c


# --------------------------------------------------------------------- inputs
def _chains(case, seed):
    """The batch of (interval, replica) chains of a Robbins-Monro case."""
    if case["kind"] == "exchange":
        w = workloads.overlapping_l4(replicas=case["replicas"], n_int=case["n_int"])
        w.n_therm, w.n_meas = case["n_therm"], case["n_meas"]
    elif case["kind"] == "rm_run":
        L, lo, de, iid, rid = [], [], [], [], []
        for g, Lg in enumerate(int(x) for x in case["Ls"].split(",")):
            dE = max(4.0, 8.0 * (Lg / 8) ** 2)
            for k, e in enumerate(workloads.place_intervals(Lg, case["n_int"], 0.58, 0.68, dE)):
                L.append(Lg), lo.append(float(e)), de.append(dE)
                iid.append(1000 * g + k), rid.append(0)
        w = workloads.Workload("run", L, lo, de, iid, rid, 0, n_therm=case["n_therm"],
                               n_meas=case["n_meas"])
    else:
        lo = workloads.place_intervals(case["L"], case["n_int"], case["e_lo"], case["e_hi"],
                                       case["dE"])
        n, r = case["n_int"], case["replicas"]
        w = workloads.Workload("rm", [case["L"]] * (n * r), [float(x) for x in np.repeat(lo, r)],
                               [case["dE"]] * (n * r), [k for k in range(n) for _ in range(r)],
                               list(range(r)) * n, 0, n_or=case["n_or"], block=case["block"],
                               n_therm=case["n_therm"], n_meas=case["n_meas"])
    w.seed = workloads.SEED_BASE + 7919 * seed
    return w


def _slopes(w, seed):
    """Slopes of a run under way: near the curve, off by a few 1e-3."""
    e = (np.asarray(w.E_lo) + 0.5 * np.asarray(w.dE)) / (6.0 * np.asarray(w.L, np.float64) ** 4)
    rng = np.random.default_rng([seed, 1])
    return -1.008 - 0.15 * (e - 0.63) + 3e-3 * rng.standard_normal(e.size)


def _links(case, seed):
    """Configurations of the ordered phase: angles of spread 0.35 around 0
    (from rougher ones a pass multiplies a rounding of 1e-7 to order 1)."""
    rng = np.random.default_rng([seed, 2])
    return rng.normal(0.0, 0.35, (case["n"], 4 * case["L"] ** 4)).astype(np.float32)


def _table(n_int, six_v, seed):
    rng = np.random.default_rng([seed, 3])
    e0, e1 = 0.59 * six_v, 0.687777 * six_v
    a = -1.0095 + 0.004 * np.sin(np.linspace(0, 3, n_int)) + 1e-4 * rng.standard_normal(n_int)
    return e0, (e1 - e0) / n_int, a


def _reweight_inputs(case, seed):
    six_v = 6.0 * 10 ** 4
    e0, de, a = _table(case["n_int"], six_v, seed)
    rng = np.random.default_rng([seed, 4])
    n = case["samples"]
    k = 2 * n // 5
    E = np.concatenate([rng.normal(0.605 * six_v, 250.0, k), rng.normal(0.645 * six_v, 250.0, k),
                        rng.uniform(0.6 * six_v, 0.65 * six_v, n - 2 * k)])
    return E[rng.permutation(n)], e0, de, a, np.linspace(1.0, 1.016, case["n_beta"])


def _recon_inputs(case, seed):
    n = case["n"]
    rng = np.random.default_rng([seed, 5])
    six_v = 6.0 * 12 ** 4
    c = np.linspace(0.59 * six_v, 0.687777 * six_v, n)
    x = np.linspace(-1.0, 1.0, n)
    a = -1.0075 - 0.004 * x - 0.002 * np.sin(2.5 * x) + 2e-5 * rng.standard_normal(n)
    return c, a, np.linspace(1.0, 1.016, case["n_beta"])


def _mlp_data(n, seed, Ls=(8, 10, 12, 14, 16)):
    rng = np.random.default_rng([seed, 6])
    L = np.repeat(np.asarray(Ls, dtype=np.float64), n)
    e = np.tile(np.linspace(0.58, 0.68, n), len(Ls))
    d = 8.0 * (L / 8.0) ** 2 / (6.0 * L ** 4)
    t = -1.008 - 0.15 * (e - 0.63) + 4.0 / L ** 4 + 2e-4 * rng.standard_normal(L.size)
    return L, e, d, t


def _mlp_params(seed):
    """Parameters of a network in training: weights of its start, small biases."""
    rng = np.random.default_rng([seed, 7])
    parts = []
    for fan, out in ((3, 64), (64, 64), (64, 64), (64, 1)):
        parts += [rng.normal(0.0, fan ** -0.5, fan * out), rng.normal(0.0, 0.05, out)]
    return np.concatenate(parts).astype(np.float32)


def prepare(case, seed):
    kind, s = case["kind"], {"case": case}
    stream = torch.cuda.current_stream().cuda_stream
    if kind in ("rm", "rm_save", "rm_run", "exchange"):
        w = _chains(case, seed)
        s["w"], s["n"] = w, 0
        s["batch"] = llr.Batch.from_workload(w, stream=stream)
        if not case.get("fast", True):
            s["batch"].set_kernel_config(256, False)
        s["a"] = _slopes(w, seed)
        if kind == "rm_run":
            s["a"] = torch.tensor(s["a"], dtype=torch.float64, device="cuda")
            s["hist"] = torch.empty((case["n_steps"], w.n_lattices), dtype=torch.float64,
                                    device="cuda")
    elif kind == "muca":
        L, n = case["L"], case["chains"]
        e0, de, a = _table(case["n_int"], 6.0 * L ** 4, seed)
        span = case["n_int"] * de
        w = workloads.Workload("muca", [L] * n, [e0] * n, [span] * n, list(range(n)), [0] * n,
                               workloads.SEED_BASE + 7919 * seed)
        s["batch"] = llr.Batch.from_workload(w, stream=stream)
        s["batch"].set_muca_weight(e0, de, a, float(a.mean()))
    elif kind in ("or_pass", "load"):
        L, n = case["L"], case["n"]
        six_v = 6.0 * L ** 4   # a window that holds every energy
        s["batch"] = llr.Batch([L] * n, [-1.1 * six_v] * n, [2.2 * six_v] * n, list(range(n)),
                               [0] * n, workloads.SEED_BASE + seed, stream=stream)
        s["links"] = _links(case, seed)
        if kind == "or_pass":
            for i in range(n):
                s["batch"].set_links(i, s["links"][i])
    elif kind == "recon":
        s["c"], s["a"], s["betas"] = _recon_inputs(case, seed)
    elif kind == "reweight":
        s["E"], s["e0"], s["de"], s["a"], s["betas"] = _reweight_inputs(case, seed)
    elif kind == "mlp_fit":
        L, e, d, t = _mlp_data(case["n"], seed)
        s["data"] = dict(L=L, e6v=e, dE6v=d, a=t)
        rng = np.random.default_rng([seed, 8])
        s["target"] = (np.full(case["n_pred"], 20.0), rng.uniform(0.58, 0.68, case["n_pred"]),
                       np.full(case["n_pred"], 50.0 / (6.0 * 20 ** 4)))
        s["seed"] = 3 + seed
    else:
        s["x"] = _mlp_data(case["n"], seed)
        s["net"] = llr.MLP(seed=seed, stream=stream)
        s["net"].set_norm([1e-4, 0.63, 1.5e-4], [8e-5, 0.03, 9e-5])
        s["net"].set_params(_mlp_params(seed))
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind in ("rm", "rm_save", "exchange"):
        b = s["batch"]
        s["a"], mean = b.rm_step(s["a"], case["n_therm"], case["n_meas"], 20 + s["n"])
        out = {"a": s["a"], "mean": mean}
        if kind == "exchange":
            pairs = workloads.exchange_pairs(s["w"], s["n"])
            out["accepted"] = b.replica_exchange(pairs, s["a"], s["n"]).astype(np.int32)
        s["n"] += 1
        out["E"] = b.tracked_energy()
        if kind == "rm_save":
            out["state"] = np.frombuffer(b.save_state(), dtype=np.uint8)
        elif kind == "exchange":
            out["links"] = np.concatenate([b.get_links(i) for i in range(b.n)])
        else:
            out["links0"] = b.get_links(0)
        return out
    if kind == "rm_run":
        s["batch"].rm_run(s["a"], case["n_therm"], case["n_meas"], 20, case["n_steps"], s["hist"])
        return {"a": s["a"], "hist": s["hist"], "E": s["batch"].tracked_energy()}
    if kind == "muca":
        E = s["batch"].muca_sweep(case["sweeps"])
        return {"E": E, "links0": s["batch"].get_links(0)}
    if kind == "or_pass":
        b = s["batch"]
        b.single_pass(1)
        return {"links": np.stack([b.get_links(i) for i in range(b.n)])}
    if kind == "load":
        b = s["batch"]
        for i in range(b.n):
            b.set_links(i, s["links"][i])
        E = b.energy()
        return {"E": E, "tracked": b.tracked_energy(),
                "links": np.stack([b.get_links(i) for i in range(b.n)])}
    if kind == "recon":
        ln = llr.reconstruct_lnrho(s["c"], s["a"])
        lnz, e1, e2 = llr.observables(s["c"], s["a"], s["betas"])
        beta_c, cv = llr.cv_peak(s["c"], s["a"], 1.0, 1.016, n_grid=case["n_grid"], tol=1e-10)
        return {"lnrho": ln, "lnZ": lnz, "E": e1, "E2": e2, "beta_c": beta_c, "cv": cv}
    if kind == "reweight":
        e1, e2 = llr.muca_reweight(s["E"], s["e0"], s["de"], s["a"], s["betas"])
        beta_c, cv = llr.muca_cv_peak(s["E"], s["e0"], s["de"], s["a"], 1.0, 1.016,
                                      n_grid=case["n_grid"], tol=1e-7)
        return {"E": e1, "E2": e2, "beta_c": beta_c, "cv": cv}
    if kind == "mlp_fit":
        net, eps, loss = warmstart.fit_network(s["data"], epochs=case["epochs"], seed=s["seed"])
        with net:
            return {"params": net.get_params(), "loss": loss, "eps": eps,
                    "a": net.predict(*s["target"])}
    g, loss = s["net"].grad(*s["x"])
    return {"grad": g, "loss": loss, "a": s["net"].predict(*s["x"][:3])}


# ----------------------------------------------------------------------- work
def work(case):
    kind = case["kind"]
    if kind in ("rm", "rm_save", "rm_run", "exchange", "muca"):
        if kind == "rm_run":
            links = sum(4 * int(x) ** 4 for x in case["Ls"].split(",")) * case["n_int"]
            sweeps, n_or = (case["n_therm"] + case["n_meas"]) * case["n_steps"], 4
        elif kind == "exchange":
            links = 4 * 4 ** 4 * case["n_int"] * case["replicas"]
            sweeps, n_or = case["n_therm"] + case["n_meas"], 4
        elif kind == "muca":
            links, sweeps, n_or = 4 * case["L"] ** 4 * case["chains"], case["sweeps"], 4
        else:
            links = 4 * case["L"] ** 4 * case["n_int"] * case["replicas"]
            sweeps, n_or = case["n_therm"] + case["n_meas"], case["n_or"]
        return {"bytes": 8.0 * links, "flops": links * sweeps * _sweep_flops(n_or)}
    if kind in ("or_pass", "load"):
        links = 4 * case["L"] ** 4 * case["n"]
        if kind == "or_pass":
            return {"bytes": 8.0 * links, "flops": FLOPS_OR * links}
        return {"bytes": 8.0 * links, "flops": 1.5 * FLOPS_PLAQUETTE * links}
    if kind == "recon":
        n, evals = case["n"], case["n_beta"] + case["n_grid"] + 40
        return {"bytes": 24.0 * n + 32.0 * case["n_beta"], "flops": FLOPS_MOMENT * n * evals}
    if kind == "reweight":
        n, evals = case["samples"], case["n_beta"] + case["n_grid"] + 18
        return {"bytes": 16.0 * n, "flops": FLOPS_MOMENT * n * evals}
    n = 5 * case["n"]
    if kind == "mlp_fit":   # the held-out training sees four of the five volumes
        steps = case["epochs"] * (n + 4 * n // 5)
        return {"bytes": 32.0 * n + 4.0 * N_PARAMS,
                "flops": 6.0 * N_PARAMS * steps + 2.0 * N_PARAMS * case["n_pred"]}
    return {"bytes": 40.0 * n + 8.0 * N_PARAMS, "flops": 8.0 * N_PARAMS * n}


# ---------------------------------------------------------------------- exact
def exact(case, seed):
    kind = case["kind"]
    if kind == "or_pass":
        return {"links": np.stack([_reflect(x, case["L"]) for x in _links(case, seed)])}
    if kind == "load":
        x = _links(case, seed)
        E = np.array([_energy(v, case["L"]) for v in x])
        return {"E": E, "tracked": E, "links": x.astype(np.float64)}
    if kind == "recon":
        c, a, betas = _recon_inputs(case, seed)
        c, a = c.astype(np.longdouble), a.astype(np.longdouble)
        ln = np.concatenate([[0.0], np.cumsum(0.5 * np.diff(c) * (a[1:] + a[:-1]))])
        w = (c[-1] - c[0]) / (c.size - 1)

        def moments(beta):
            x = ln + np.longdouble(beta) * c
            e = np.exp(x - x.max())
            return x.max() + np.log(w * e.sum()), (c * e).sum() / e.sum(), \
                (c * c * e).sum() / e.sum()

        m = np.array([moments(b) for b in betas])
        beta_c, cv = _peak(lambda b: _central(c, ln + np.longdouble(b) * c), case["n_grid"], 1e-10)
        return {"lnrho": ln.astype(np.float64), "lnZ": m[:, 0].astype(np.float64),
                "E": m[:, 1].astype(np.float64), "E2": m[:, 2].astype(np.float64),
                "beta_c": beta_c, "cv": cv}
    if kind == "reweight":
        E, e0, de, a, betas = _reweight_inputs(case, seed)
        n = a.size
        edge = np.concatenate([[0.0], np.cumsum(a * de)])
        k = np.clip(np.floor((E - e0) / de), 0, n - 1).astype(np.int64)
        lr = edge[k] + a[k] * (E - (e0 + k * de))
        d = E - e0

        def moments(beta):
            x = beta * d + lr
            w = np.exp(x - x.max())
            u = (w * d).sum() / w.sum()
            return u, (w * (d - u) ** 2).sum() / w.sum()

        m = np.array([moments(b) for b in betas])
        e1 = e0 + m[:, 0]
        beta_c, cv = _peak(lambda b: moments(b)[1], case["n_grid"], 1e-7)
        return {"E": e1, "E2": e1 * e1 + m[:, 1], "beta_c": beta_c, "cv": cv}
    if kind == "mlp_grad":
        L, e, d, t = _mlp_data(case["n"], seed)
        return _mlp_exact(_mlp_params(seed).astype(np.float64), L, e, d, t)
    return None   # chains and trainings: the outcome of many dependent roundings


def _reflect(theta, L):
    """One overrelaxation pass in 64 bits: x3 slab by slab, in each the classes
    (direction, parity); theta' = -theta - 2 arg S, wrapped to [-pi, pi)."""
    th = theta.astype(np.float64).reshape(4, L, L, L, L)   # [mu][x3][x2][x1][x0]
    x3, x2, x1, x0 = np.indices((L, L, L, L))
    parity = (x3 + x2 + x1 + x0) & 1
    axis = (3, 2, 1, 0)                                    # array axis of direction mu

    def rows(t):
        return np.arange(t - 1, t + 2) % L

    for t in range(L):
        for cls in range(8):
            mu, p = cls >> 1, cls & 1
            local = th[:, rows(t)]                         # slabs t - 1, t, t + 1

            def at(nu, *steps):
                v = local[nu]
                up = 1
                for direction, sign in steps:
                    if direction == 3:
                        up += sign
                    else:
                        v = np.roll(v, -sign, axis=axis[direction])
                return v[up]

            S = np.zeros((L, L, L), dtype=np.complex128)
            for nu in range(4):
                if nu == mu:
                    continue
                S += np.exp(1j * (at(nu, (mu, 1)) - at(mu, (nu, 1)) - at(nu)))
                S += np.exp(1j * (at(nu, (nu, -1)) - at(nu, (nu, -1), (mu, 1))
                                  - at(mu, (nu, -1))))
            new = -th[mu, t] - 2.0 * np.angle(S)
            new -= 2.0 * np.pi * np.floor((new + np.pi) / (2.0 * np.pi))
            sel = parity[t] == p
            th[mu, t][sel] = new[sel]
    return th.reshape(-1)


def _energy(theta, L):
    th = theta.astype(np.float64).reshape(4, L, L, L, L)
    axis = (3, 2, 1, 0)
    E = 0.0
    for mu in range(4):
        for nu in range(mu + 1, 4):
            E += np.cos(th[mu] + np.roll(th[nu], -1, axis=axis[mu])
                        - np.roll(th[mu], -1, axis=axis[nu]) - th[nu]).sum()
    return E


def _central(c, x):
    w = np.exp(x - x.max())
    w /= w.sum()
    u = (w * c).sum()
    return (w * (c - u) ** 2).sum()


def _peak(f, n_grid, tol, lo=1.0, hi=1.016):
    grid = np.linspace(lo, hi, n_grid)
    i = int(np.argmax([f(b) for b in grid]))
    lo, hi = grid[max(i - 1, 0)], grid[min(i + 1, n_grid - 1)]
    g = (math.sqrt(5.0) - 1.0) / 2.0
    x1, x2 = hi - g * (hi - lo), lo + g * (hi - lo)
    f1, f2 = f(x1), f(x2)
    while hi - lo > tol:
        if f1 < f2:
            lo, x1, f1 = x1, x2, f2
            x2 = lo + g * (hi - lo)
            f2 = f(x2)
        else:
            hi, x2, f2 = x2, x1, f1
            x1 = hi - g * (hi - lo)
            f1 = f(x1)
    b = 0.5 * (lo + hi)
    return float(b), float(f(b))


def _mlp_exact(P, L, e, d, t):
    shapes = ((3, 64), (64,), (64, 64), (64,), (64, 64), (64,), (64, 1), (1,))
    p, k = [], 0
    for sh in shapes:
        p.append(P[k:k + int(np.prod(sh))].reshape(sh))
        k += int(np.prod(sh))
    raw = np.stack([1.0 / L ** 4, e, d], axis=1)
    H = (raw - np.array([1e-4, 0.63, 1.5e-4])) / np.array([8e-5, 0.03, 9e-5])
    erf = np.vectorize(math.erf)
    acts, zs = [H], []
    for layer in range(4):
        z = acts[-1] @ p[2 * layer] + p[2 * layer + 1]
        zs.append(z)
        acts.append(0.5 * z * (1.0 + erf(z / math.sqrt(2.0))) if layer < 3 else z)
    y = acts[-1][:, 0]
    dz = (2.0 * (y - t) / t.size)[:, None]
    grads = [None] * 8
    for layer in (3, 2, 1, 0):
        grads[2 * layer], grads[2 * layer + 1] = acts[layer].T @ dz, dz.sum(axis=0)
        if layer:
            z = zs[layer - 1]
            dz = (dz @ p[2 * layer].T) * (0.5 * (1.0 + erf(z / math.sqrt(2.0)))
                                          + z * np.exp(-0.5 * z * z) / math.sqrt(2.0 * math.pi))
    return {"grad": np.concatenate([g.reshape(-1) for g in grads]),
            "loss": float(np.mean((y - t) ** 2)), "a": y}
