"""Cases that time this library as its users call it: a batch of wires in, currents (or
gradients, conductances, tables) out, through the public calls of paper_1805_10164_gb300.

Every case is one whole call sequence of a user's program on the configurations of
``paper_1805_10164_gb300.inputs`` (seeded synthetic wires), from the 20-site chain whose time
is launches and copies to the 64,000-site wire whose time is block products.
"""
import math
from types import SimpleNamespace

import numpy as np
import torch

from paper_1805_10164_gb300 import autograd, inputs, negf

# what a case's "kind" stands for
#   run       one batch of host wires built, walked and reduced once (negf_run + negf_current)
#   plan      a fixed batch relaunched many times (captured plan over device-resident wires)
#   tables    tables and their weights exported for another program
#   gradient  one training iteration: forward and backward of the current through autograd
#   thermal   linear conductance with energies drawn from the thermal window
#   inelastic walks whose energy changes at every probe


def listed():
    return [
        # one 20-site chain at one energy in double precision: the smallest thing a user runs,
        # a launch-and-copy-bound call
        dict(name="chain_1x20_fp64", kind="run", W=1, L=20, n_energy=1, n_wires=1, eta=0.1,
             disorder=0.5, e_lo=0.25, e_hi=0.75, walkers=100_000, precision="fp64"),
        # the ordinary wire: 500 sites, 64 energies over the band, 1e6 walkers each, as a
        # captured plan that is launched again and again
        dict(name="wire_10x50_plan", kind="plan", W=10, L=50, n_energy=64, n_wires=1, eta=0.05,
             disorder=1.0, e_lo=-3.5, e_hi=3.5, walkers=1_000_000, precision="fp32"),
        # the same wire with the tables in double precision, as the paper computes them
        dict(name="wire_10x50_fp64", kind="run", W=10, L=50, n_energy=64, n_wires=1, eta=0.05,
             disorder=1.0, e_lo=-3.5, e_hi=3.5, walkers=1_000_000, precision="fp64"),
        # a disorder / size study: wires of uneven width and length in one call
        dict(name="uneven_batch", kind="run", W=0, L=0, n_energy=32, n_wires=40, eta=0.0,
             disorder=1.0, e_lo=-3.5, e_hi=3.5, walkers=1_000_000, precision="fp32"),
        # the widest and longest wire (weak scattering, two-level tables), a few of its energies
        dict(name="weak_64x1000_plan", kind="plan", W=64, L=1000, n_energy=4, n_wires=1,
             eta=0.005, disorder=0.5, e_lo=-3.5, e_hi=3.5, walkers=32_000_000,
             precision="fp32"),
        # a wide wire of medium length, one call over host arrays
        dict(name="wide_64x100", kind="run", W=64, L=100, n_energy=8, n_wires=1, eta=0.005,
             disorder=0.5, e_lo=-3.5, e_hi=3.5, walkers=1_000_000, precision="fp32"),
        # a multi-orbital film: 10 atoms of 4 orbitals per slice, 4 k-points
        dict(name="film_40x50_4k", kind="run", W=40, L=50, n_energy=4, n_wires=4, eta=0.1,
             disorder=0.5, e_lo=-1.5, e_hi=2.5, walkers=200_000, precision="fp32",
             film=True),
        # one training iteration of the differentiation case (1600 onsite energies and rates)
        dict(name="gradient_16x100", kind="gradient", W=16, L=100, n_energy=16, n_wires=1,
             eta=0.05, disorder=1.0, e_lo=-3.5, e_hi=3.5, walkers=1_000_000,
             precision="fp32"),
        # the inner loop of fitting a small wire: many short iterations
        dict(name="gradient_4x20", kind="gradient", W=4, L=20, n_energy=8, n_wires=1, eta=0.1,
             disorder=1.0, e_lo=-2.9, e_hi=2.9, walkers=100_000, precision="fp32"),
        # linear conductance over the thermal window on an adaptive energy grid
        dict(name="thermal_10x50", kind="thermal", W=10, L=50, n_energy=0, n_wires=1, eta=0.05,
             disorder=1.0, e_lo=0.0, e_hi=0.0, walkers=16_000_000, precision="fp32"),
        # inelastic probes on the ordinary wire
        dict(name="inelastic_10x50", kind="inelastic", W=10, L=50, n_energy=64, n_wires=1,
             eta=0.05, disorder=1.0, e_lo=-3.5, e_hi=3.5, walkers=1_000_000,
             precision="fp32"),
        # the Step 6' weights themselves, read back by another program
        dict(name="tables_10x50", kind="tables", W=10, L=50, n_energy=8, n_wires=1, eta=0.05,
             disorder=1.0, e_lo=-3.5, e_hi=3.5, walkers=0, precision="fp32"),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["run", "run", "run", "plan", "tables", "gradient", "thermal", "inelastic"])
    case = dict(kind=kind, n_wires=1, eta=math.exp(rng.uniform(math.log(0.005), math.log(0.2))),
                disorder=rng.choice([0.5, 1.0]), e_lo=-3.47, e_hi=3.49,
                walkers=_log_int(rng, 20_000, 1_000_000), precision="fp32")
    if kind in ("run", "plan"):
        W = rng.choice([rng.randint(1, 16), rng.randint(4, 32), rng.randint(33, 64)])
        L = _log_int(rng, 2, 300)
        case["precision"] = "fp64" if W <= 16 and rng.random() < 0.3 else "fp32"
        case["film"] = W % 4 == 0 and rng.random() < 0.3
        n = _log_int(rng, 1, 64)
        case["n_wires"] = 4 if case["film"] else rng.choice([1, 1, 3])
    elif kind == "tables":
        W, L, n = rng.randint(1, 16), _log_int(rng, 5, 60), rng.randint(1, 8)
        case["precision"] = rng.choice(["fp32", "fp64"])
        case["walkers"] = 0
    elif kind == "gradient":
        W, L, n = rng.randint(2, 24), _log_int(rng, 5, 100), rng.randint(2, 16)
    else:
        W, L, n = rng.randint(2, 16), _log_int(rng, 5, 80), rng.randint(8, 64)
        case["eta"] = max(case["eta"], 0.02)
        if kind == "thermal":
            case.update(n_energy=0, e_lo=0.0, e_hi=0.0)
    # block products stay well below the largest listed case's, and two-level table memory small
    most = 1e11 if case["precision"] == "fp32" else 4e9
    while W * L > 16_384 or 8.0 * W ** 3 * L * L * n * case["n_wires"] > most:
        if n > 1:
            n = max(1, n // 2)
        else:
            L = max(2, L // 2)
    case.update(W=W, L=L, n_energy=0 if kind == "thermal" else n)
    return case


# ---------------------------------------------------------------- inputs

MU, KT = (3.5, -3.5), 0.025     # the bias window of the wires' currents
THERMAL = dict(n_init=9, tol=0.05, max_points=257)
SIGMA_E = 0.1                   # width of the inelastic probes' energy exchange
MAX_STEPS = 1 << 20


def _wires(case, seed):
    rng = np.random.default_rng(seed)
    E, wE = inputs.midpoint_grid(case["e_lo"], case["e_hi"], max(1, case["n_energy"]))
    if case.get("film"):
        atoms = case["W"] // 4
        base = inputs.sp3_wire(seed, atoms, case["L"], n_energy=case["n_energy"],
                               eta=case["eta"], disorder=case["disorder"], e_lo=case["e_lo"],
                               e_hi=case["e_hi"])
        return inputs.film_kpoints(base, 0.3, case["n_wires"])
    if case["W"] == 0:
        # uneven wires: W uniform in 4..32, L uniform in 20..200, eta log-uniform
        out = []
        for _ in range(case["n_wires"]):
            W, L = int(rng.integers(4, 33)), int(rng.integers(20, 201))
            eta = float(np.exp(rng.uniform(np.log(0.01), np.log(0.2))))
            out.append(inputs.random_wire(rng, W, L, 1.0, case["disorder"], eta, E, wE))
        return out
    return [inputs.random_wire(rng, case["W"], case["L"], 1.0, case["disorder"], case["eta"], E,
                               wE) for _ in range(case["n_wires"])]


def _on_device(w):
    t = {k: None if getattr(w, k) is None else torch.from_numpy(np.ascontiguousarray(
        getattr(w, k))).cuda() for k in ("onsite", "eta", "energy", "energy_weight", "slice_h")}
    return SimpleNamespace(W=w.W, L=w.L, t=w.t, lead_model=w.lead_model,
                           gamma_lead=w.gamma_lead, **t)


class _State:
    """A context, and the plan a program keeps with it; given back when the state goes."""

    def __init__(self, case, seed):
        self.case, self.seed, self.plan = case, seed, None
        self.ctx = negf.negf_create(torch.cuda.current_device())

    def __del__(self):
        if self.plan is not None:
            negf.negf_plan_destroy(self.plan)
        negf.negf_destroy(self.ctx)


def prepare(case, seed):
    s = _State(case, seed)
    s.wires = _wires(case, seed)
    s.n_tasks = sum(len(w.energy) for w in s.wires)
    kind = case["kind"]
    if kind == "plan":
        s.dev = [_on_device(w) for w in s.wires]
        # a wave of one task at a time where one task's tables are gigabytes
        one_by_one = case["W"] * case["L"] > 32_768
        s.plan = negf.negf_plan_create(s.ctx, s.dev, 0, case["walkers"], *MU, KT,
                                       precision=case["precision"], memspace="device",
                                       max_steps=MAX_STEPS,
                                       tasks_per_wave=1 if one_by_one else 0)
    elif kind == "gradient":
        w = s.wires[0]
        s.onsite = torch.from_numpy(w.onsite).cuda().requires_grad_()
        s.eta = torch.from_numpy(w.eta).cuda().requires_grad_()
        s.spec = autograd.CurrentSpec(
            W=w.W, L=w.L, t=w.t, energy=torch.from_numpy(w.energy).cuda(),
            energy_weight=torch.from_numpy(w.energy_weight).cuda(), mu_p=MU[0], mu_q=MU[1],
            kT=KT, walkers_per_task=case["walkers"], seed=seed, max_steps=MAX_STEPS,
            precision=case["precision"])
    elif kind == "thermal":
        w = s.wires[0]
        w.energy = negf.negf_thermal_grid(s.ctx, w, -8 * KT, 8 * KT, precision=case["precision"],
                                          **THERMAL)
        w.energy_weight = np.ones_like(w.energy)
        s.dev = [_on_device(w)]
    elif kind == "inelastic":
        s.dev = [_on_device(w) for w in s.wires]
    return s


# ---------------------------------------------------------------- one pass

def run(s):
    case, ctx = s.case, s.ctx
    kind = case["kind"]
    if kind == "run":
        tables, tally = negf.negf_run(ctx, s.wires, 0, s.seed, case["walkers"],
                                      precision=case["precision"], max_steps=MAX_STEPS)
        res = negf.negf_current(ctx, tables, tally, *MU, KT)
        out = dict(I=res["I"], se=res["se"], T=res["T"], T_se=res["T_se"],
                   counts=negf.negf_tally_counts(ctx, tally, s.n_tasks))
        if s.n_tasks == 1:
            out["c"] = negf.negf_get_task_info(ctx, tables, 0)["c"]
        negf.negf_tally_free(tally)
        negf.negf_tables_free(tables)
        return out
    if kind == "plan":
        negf.negf_plan_launch(ctx, s.plan, s.seed)
        res = negf.negf_plan_result(ctx, s.plan)
        return {k: res[k] for k in ("I", "se", "T", "T_se", "counts")}
    if kind == "gradient":
        s.onsite.grad = s.eta.grad = None
        I, se = autograd.current(s.onsite, s.eta, ctx, s.spec)
        I.backward()
        return dict(I=I.detach(), se=se, d_onsite=s.onsite.grad, d_eta=s.eta.grad)
    if kind == "thermal":
        tables = negf.negf_build_tables(ctx, s.dev, precision=case["precision"],
                                        memspace="device")
        res = negf.negf_walk_thermal(ctx, tables, 0, 0, s.seed, case["walkers"], 0.0, KT,
                                     max_steps=MAX_STEPS)
        negf.negf_tables_free(tables)
        return {k: res[k] for k in ("G", "se", "window", "mean_steps", "absorbed", "closed")}
    if kind == "inelastic":
        tables = negf.negf_build_tables(ctx, s.dev, precision=case["precision"],
                                        memspace="device")
        tally = negf.negf_walk_inelastic(ctx, tables, 0, s.seed, case["walkers"], SIGMA_E,
                                         max_steps=MAX_STEPS)
        res = negf.negf_current(ctx, tables, tally, *MU, KT)
        out = dict(I=res["I"], se=res["se"], T=res["T"], T_se=res["T_se"],
                   counts=negf.negf_tally_counts(ctx, tally, s.n_tasks))
        negf.negf_tally_free(tally)
        negf.negf_tables_free(tables)
        return out
    # tables: every energy's weights, row sums, mode weights and Tr[Gamma_p A]
    tables = negf.negf_build_tables(ctx, s.wires, precision=case["precision"], keep_weights=True)
    out = {}
    for what in ("weights", "rowsum", "mode_weights"):
        out[what] = np.stack([negf.negf_export_tables(ctx, tables, t, what)
                              for t in range(s.n_tasks)])
    out["c"] = np.stack([negf.negf_get_task_info(ctx, tables, t)["c"]
                         for t in range(s.n_tasks)])
    negf.negf_tables_free(tables)
    return out


# ---------------------------------------------------------------- what a pass cannot do without

def work(case):
    """Bytes: the wires in, the results out, and one 8-byte table entry per draw of the shortest
    walk (an injection and one transition).  Flops: the block products of one task's columns
    (towards one side; the other by symmetry) and of its two sweeps, in real operations."""
    if case["W"] == 0:
        # mean over the uniform ranges W in 4..32, L in 20..200
        w3 = sum(w ** 3 for w in range(4, 33)) / 29.0
        l2 = sum(l * l for l in range(20, 201)) / 181.0
        sites, products, sweeps = 18.0 * 110.0, w3 * l2 / 2, 2 * w3 * 110.0
    else:
        W, L = case["W"], case["L"]
        sites, products, sweeps = W * L, W ** 3 * L * (L - 1) / 2, 2 * W ** 3 * L
    grid = case["n_energy"] or THERMAL["n_init"]
    tasks = grid * case["n_wires"]
    walks = case["walkers"] * (1 if case["kind"] == "thermal" else tasks)
    out = 8.0 * 8 * tasks
    if case["kind"] == "tables":
        rows, K = sites + 2 * case["W"], sites + 2
        out = 8.0 * tasks * (rows * K + rows)
    elif case["kind"] == "gradient":
        out += 8.0 * 2 * sites
        products *= 3        # the columns, and their elimination back
    return dict(bytes=16.0 * sites * case["n_wires"] + out + 16.0 * walks,
                flops=8.0 * tasks * (products + sweeps))


# ---------------------------------------------------------------- the same in 64 bits

def _strip_modes(W, E, t):
    """Transverse modes of a clean square-lattice strip and their self-energies."""
    a = np.arange(1, W + 1)
    phi = math.sqrt(2.0 / (W + 1)) * np.sin(np.pi * np.outer(a, a) / (W + 1))
    e = E + 2.0 * t * np.cos(np.pi * a / (W + 1))
    inside = np.abs(e) < 2.0 * t
    r = np.sqrt(np.abs(4.0 * t * t - e * e))
    sig = np.where(inside, 0.5 * e - 0.5j * r, 0.5 * (e - np.sign(e) * r))
    return phi, sig, np.where(inside, r, 0.0)


def _exact_task(w, E):
    """Weights [rows, K], row sums, mode weights [2, W] and c [2] of one energy by dense
    inversion."""
    W, L, n = w.W, w.L, w.W * w.L
    H = np.diag(w.onsite.reshape(-1).astype(float))
    i = np.arange(n)
    for step, ok in ((1, (i % W) != W - 1), (W, i < n - W)):
        j = i[ok]
        H[j, j + step] -= w.t
        H[j + step, j] -= w.t
    phi, sig, gam = _strip_modes(W, E, w.t)
    M = E * np.eye(n) - H + 0.5j * np.diag(w.eta.reshape(-1))
    ends = (slice(0, W), slice(n - W, n))
    for p in ends:
        M[p, p] -= phi @ np.diag(sig) @ phi.T
    G = np.linalg.inv(M)
    gphi = [G[:, p] @ phi for p in ends]                        # G Phi of each lead
    cols = np.concatenate([G, gphi[0], gphi[1]], axis=1)        # one column per table row
    site = w.eta.reshape(-1, 1) * np.abs(cols) ** 2
    lead = [np.sum(gam[:, None] * np.abs(phi.T @ cols[p]) ** 2, axis=0) for p in ends]
    A = -2.0 * np.concatenate([np.diag(G).imag] + [np.einsum("ab,ab->b", phi, g[p].imag)
                                                   for g, p in zip(gphi, ends)])
    mode = np.stack([gam * A[n:n + W], gam * A[n + W:]])
    weights = np.concatenate([site, lead[0][None], lead[1][None]], axis=0).T
    return weights, A, mode, mode.sum(axis=1)


def exact(case, seed):
    """Tables, row sums, mode weights and Tr[Gamma_p A] by dense inversion; sampled currents and
    gradients have no exact value on a given random stream."""
    one_task = case["kind"] == "run" and case["n_energy"] * case["n_wires"] == 1
    if case.get("film") or not (case["kind"] == "tables" or one_task) or case["W"] * case["L"] > 1024:
        return None
    w = _wires(case, seed)[0]
    tasks = [_exact_task(w, E) for E in w.energy]
    if one_task:
        return dict(I=None, se=None, T=None, T_se=None, counts=None, c=tasks[0][3])
    return dict(weights=np.stack([t[0].reshape(-1) for t in tasks]),
                rowsum=np.stack([t[1] for t in tasks]),
                mode_weights=np.stack([t[2].reshape(-1) for t in tasks]),
                c=np.stack([t[3] for t in tasks]))
