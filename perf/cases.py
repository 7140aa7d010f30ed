"""The work that a user of the library has it do, as measurable cases.

A case is a dict of plain values; ``kind`` says which entry points it goes
through:

``scan``     one or more transformations l -> l+1 of one lattice shape in a
             jarzynski_run_batch call, then the FP64 estimate of each l: the
             c-function scan.  ``host`` puts the work arrays in host memory.
``segment``  one transformation in two protocol segments with its spins and
             work kept on the device between them (checkpoint / resume).
``plan``     an uneven batch of several lattice shapes, replayed from its
             persistent plan, with the batched estimates.
``serve``    a burst of mixed jobs submitted to a running server and waited
             for, with their work arrays fetched.
``reduce``   the estimator alone on stored work values.

Lattice sizes, couplings, protocol lengths and l ranges are those of the
library's workloads and of its benchmark options, with fewer trajectories or
shorter protocols where a full run takes longer than two seconds.
"""
import math
import random

import numpy as np
import torch

import paper_2304_03311_gb300 as jz
from paper_2304_03311_gb300.workloads import BETA_C_2D, BETA_C_3D, BETA_3D_CONFIG

# Counted integer operations of one Metropolis spin update (2D, 3D) and of one
# Swendsen-Wang site visit: random numbers, local field, acceptance / bonds.
OPS_UPDATE = {2: 32, 3: 36}
OPS_CLUSTER = 104


def _scan(**kw):
    c = dict(kind="scan", d=2, L=64, L_t=64, beta=BETA_C_2D, l0=0, l_step=1, n_l=1, n_step=1000,
             n_sweep=1, n_therm=1000, n_traj=1024, direction=1, update=0, therm_update=0,
             n_replica=2, whole=False, protocol=1, host=False)
    c.update(kw)
    return c


def listed():
    return [
        # the estimator on the work values of one l of the 2D L = 64 scan: the
        # smallest call, made once per l of every scan
        dict(name="reduce_16384", kind="reduce", n=16384, n_step=1000, beta=BETA_C_2D,
             direction=1, bins=32, mean=2.0, width=1.5),
        # one small transformation with its work in host memory (the 2D L = 16
        # workload as it is): a latency-bound call
        _scan(name="single_2d_L16", L=16, L_t=16, l0=4, n_step=200, n_traj=1000, host=True),
        # the 2D L = 64 c-function scan, every l, at a sixteenth of its trajectories
        _scan(name="scan_2d_L64", n_l=31, n_sweep=2),
        # the 3D slab scan at a quarter of its trajectories
        _scan(name="scan_3d_L16", d=3, L=16, L_t=16, beta=BETA_3D_CONFIG, l0=1, n_l=8,
              n_step=2000),
        # the paper's own update, clusters throughout, on the 2D L = 64 scan
        _scan(name="clusters_2d_L64", n_l=31, n_step=200, n_therm=100, n_traj=64, update=1),
        # the unbiased scan that the benchmark recommends: a cluster start of
        # 100 sweeps, then the Metropolis protocol
        _scan(name="cluster_start_2d_L64", n_l=31, n_step=500, n_sweep=2, n_therm=100,
              n_traj=512, therm_update=1),
        # the paper's largest 2D lattice, L_t = 8 L, every 16th l
        _scan(name="tall_2d_L128", L=128, L_t=1024, l0=1, l_step=16, n_l=8, n_step=500,
              n_therm=500, n_traj=64),
        # the paper's smaller 3D lattice, L_t = 4 L: rows that do not fill
        # whole spin words, and the reverse transformation
        _scan(name="slab_3d_L24", d=3, L=24, L_t=96, beta=BETA_C_3D, l0=1, l_step=3, n_l=4,
              n_step=600, n_therm=400, n_traj=256, direction=-1),
        # the paper's largest 3D lattice, L_t = 4 L, from a cluster start: both
        # updates on states beyond shared memory
        _scan(name="slab_3d_L48", d=3, L=48, L_t=192, beta=BETA_C_3D, l0=2, l_step=3, n_l=2,
              n_step=200, n_therm=20, n_traj=128, therm_update=1),
        # three replicas, a whole cut, on ragged rows, checkpointed halfway
        dict(_scan(name="segment_2d_L40", L=40, L_t=40, l0=12, n_step=400, n_therm=200,
                   n_traj=2048, n_replica=3, whole=True), kind="segment"),
        # the uneven batch over its nine lattice shapes, three l values each
        dict(name="plan_uneven", kind="plan", mix=0, n_l=3, traj_lo=6, traj_hi=9, step_lo=200,
             step_octaves=3, n_therm=300),
        # a burst of the served stream's jobs (2D and 3D, L from 8 to 256,
        # three temperatures), all at once
        dict(name="serve_burst", kind="serve", mix=0, n_jobs=32, traj_lo=7, traj_hi=9, n_step=200,
             n_therm=200, inflight=16),
    ]


# ------------------------------------------------------------------- jobs --
def _mix(case):
    """(d, L, L_t, beta, l, n_step, n_traj) of the jobs of a plan or a burst:
    the case's mix number draws them."""
    rng = np.random.default_rng(case["mix"])
    out = []
    if case["kind"] == "plan":
        shapes = [(2, L) for L in (32, 48, 64, 96, 128)] + [(3, L) for L in (8, 12, 16, 24)]
        for d, L in shapes:
            for l in sorted(1 + rng.choice(L // 2, size=case["n_l"], replace=False)):
                out.append((d, L, L, BETA_C_2D if d == 2 else BETA_C_3D, int(l),
                            int(case["step_lo"] * 2 ** rng.integers(0, case["step_octaves"])),
                            int(2 ** rng.integers(case["traj_lo"], case["traj_hi"] + 1))))
    else:
        for _ in range(case["n_jobs"]):
            d = int(rng.integers(2, 4))
            L = int(2 * (rng.integers(16, 129) if d == 2 else rng.integers(4, 25)))
            beta = float((BETA_C_2D if d == 2 else BETA_C_3D) *
                         (0.9, 1.0, 1.1)[int(rng.integers(0, 3))])
            out.append((d, L, L, beta, int(rng.integers(1, L // 2 + 1)), case["n_step"],
                        int(2 ** rng.integers(case["traj_lo"], case["traj_hi"] + 1))))
    return out


def _cost(case):
    """(Metropolis spin updates by dimension, cluster site visits, trajectories,
    spins returned) of one pass."""
    upd = {2: 0, 3: 0}
    clu = traj = spins = 0
    if case["kind"] in ("plan", "serve"):
        for d, L, L_t, _, _, n_step, n_traj in _mix(case):
            upd[d] += n_traj * 2 * L_t * L ** (d - 1) * (case["n_therm"] + n_step)
            traj += n_traj
    elif case["kind"] != "reduce":
        d = case["d"]
        V = case["n_replica"] * case["L_t"] * case["L"] ** (d - 1)
        traj = case["n_l"] * case["n_traj"]
        prot = traj * V * case["n_step"] * case["n_sweep"]
        therm = traj * V * case["n_therm"]
        clu += (prot if case["update"] else 0) + \
            (therm if case["update"] or case["therm_update"] else 0)
        upd[d] += (0 if case["update"] else prot) + \
            (0 if case["update"] or case["therm_update"] else therm)
        spins = traj * V if case["kind"] == "segment" else 0
    return upd, clu, traj, spins


def work(case):
    if case["kind"] == "reduce":
        # one exponential (about 20 FP64 operations) and a few sums per value
        return {"bytes": 8 * case["n"], "flops": 24 * case["n"]}
    upd, clu, traj, spins = _cost(case)
    ops = sum(OPS_UPDATE[d] * u for d, u in upd.items()) + OPS_CLUSTER * clu
    return {"bytes": 8 * traj + spins, "flops": ops}


# ------------------------------------------------------------------- draw --
def _log2_int(rng, lo, hi):
    """A whole number in [lo, hi], even over its logarithm."""
    return min(hi, max(lo, int(round(2 ** rng.uniform(math.log2(lo), math.log2(hi))))))


def _even(rng, lo, hi):
    return 2 * _log2_int(rng, lo // 2, hi // 2)


def draw(rng: random.Random):
    """One more case of the listed kinds: sizes, l ranges, temperatures and
    options over their whole range, trajectories set by a cost drawn below the
    largest listed case's."""
    kind = rng.choice(["scan"] * 6 + ["segment", "plan", "serve", "reduce"])
    if kind == "reduce":
        n = _log2_int(rng, 200, 200000)
        return dict(kind=kind, n=n, n_step=_log2_int(rng, 100, 4000),
                    beta=rng.choice([BETA_C_2D, BETA_C_3D]), direction=rng.choice([1, -1]),
                    bins=rng.choice([1, 10, 32, 64]), mean=rng.uniform(0.0, 4.0),
                    width=rng.uniform(0.2, 2.0))
    if kind == "plan":
        return dict(kind=kind, mix=rng.randrange(1 << 30), n_l=rng.randint(1, 4), traj_lo=5,
                    traj_hi=rng.randint(6, 8), step_lo=rng.randint(60, 200), step_octaves=3,
                    n_therm=rng.randint(50, 300))
    if kind == "serve":
        return dict(kind=kind, mix=rng.randrange(1 << 30), n_jobs=rng.randint(3, 40), traj_lo=6,
                    traj_hi=rng.randint(7, 9), n_step=rng.randint(50, 200),
                    n_therm=rng.randint(50, 200), inflight=rng.choice([4, 16]))
    d = rng.choice([2, 2, 3])
    L = _even(rng, 10, 200) if d == 2 else _even(rng, 6, 40)
    L_t = L * rng.choice([1, 1, 1, 4, 8] if d == 2 else [1, 1, 4])
    if L_t > 1024:
        L_t = L
    beta = (BETA_C_2D if d == 2 else BETA_C_3D) * rng.choice([0.9, 1.0, 1.0, 1.0, 1.1])
    update, therm_update = rng.choice([(0, 0), (0, 0), (0, 0), (1, 0), (0, 1)])
    n_replica = rng.choice([2, 2, 2, 3, 4])
    if update and 4.75 * n_replica * L_t * L ** (d - 1) > 200000:
        L_t = L = 2 * rng.randint(4, 32 if d == 2 else 8)   # cluster states in shared memory
    whole = rng.random() < 0.2
    protocol = 2 if d == 3 and not whole and rng.random() < 0.25 else 1
    n_sweep = rng.choice([1, 1, 2])
    n_step = _log2_int(rng, 50, 1000)
    n_step += -n_step % L if protocol == 2 else 0
    n_therm = _log2_int(rng, 20, 1000) if not (update or therm_update) else rng.randint(10, 60)
    n_l = rng.randint(1, 8) if kind == "scan" else 1
    l0 = rng.randint(1, max(1, L // 2))
    l_step = rng.randint(1, 3)
    while l0 + l_step * (n_l - 1) > L - 1:
        n_l -= 1
    V = n_replica * L_t * L ** (d - 1)
    # Metropolis-equivalent updates: a cluster site visit costs about 14, and
    # about 30 on a state beyond shared memory
    per = (14 if 4.75 * V < 220000 else 30)
    per_traj = V * (n_step * n_sweep * (per if update else 1) +
                    n_therm * (per if update or therm_update else 1))
    budget = 2 ** rng.uniform(28, 37.5)
    n_traj = max(16, min(8192, int(budget / (per_traj * n_l))))
    n_traj += (n_traj > 64 and rng.random() < 0.5)
    while per_traj * n_traj * n_l > 3e11 and n_step >= 2 * max(L, 20):   # the largest lattices
        n_step //= 2
        n_step -= n_step % L if protocol == 2 else 0
        n_therm = max(10, n_therm // 2)
        per_traj = V * (n_step * n_sweep * (per if update else 1) +
                        n_therm * (per if update or therm_update else 1))
    c = _scan(d=d, L=L, L_t=L_t, beta=beta, l0=l0, l_step=l_step, n_l=n_l, n_step=n_step,
              n_sweep=n_sweep, n_therm=n_therm, n_traj=n_traj, direction=rng.choice([1, 1, -1]),
              update=update, therm_update=therm_update, n_replica=n_replica, whole=whole,
              protocol=protocol, host=rng.random() < 0.3)
    c["kind"] = kind
    if kind == "segment":
        c["host"] = False
        c["n_traj"] = min(n_traj, max(16, (1 << 28) // V))   # the spins it keeps
    return c


# ---------------------------------------------------------------- prepare --
class _State:
    """What a user's program keeps between calls; released with it."""

    def __init__(self, kind):
        self.kind = kind
        self.ctx = jz.ising_replica_init(0, 0, None)
        self.plan = self.server = None

    def __del__(self):
        try:
            if self.plan:
                jz.jz_plan_free(self.plan)
            if self.server:
                jz.jz_server_free(self.server)
            jz.ising_replica_free(self.ctx)
        except Exception:
            pass


def _work_values(case, seed):
    """Integer work values of the scale that a protocol yields: W is about
    mean +- width, and W_int = W n_step / beta, an even number."""
    g = torch.Generator().manual_seed(seed)
    w = case["mean"] + case["width"] * torch.randn(case["n"], generator=g, dtype=torch.float64)
    return 2 * torch.round(0.5 * w * case["n_step"] / case["beta"]).to(torch.int64)


def prepare(case, seed):
    s = _State(case["kind"])
    s.case = case
    if case["kind"] == "reduce":
        s.work = _work_values(case, seed).cuda()
        return s
    if case["kind"] in ("plan", "serve"):
        s.jobs = []
        for i, (d, L, L_t, beta, l, n_step, n_traj) in enumerate(_mix(case)):
            # a plan's jobs share one seed, their trajectory ranges set them apart
            own = dict(seed=seed, traj0=i << 20) if case["kind"] == "plan" else dict(
                seed=seed * 1000 + i)
            s.jobs.append(jz.make_params(d, L, L_t, beta, l, n_step, 1, n_traj,
                                         n_therm=case["n_therm"], **own))
        if case["kind"] == "plan":
            s.out = [torch.empty(p.n_traj, dtype=torch.int64, device="cuda") for p in s.jobs]
            s.est = torch.empty(len(s.jobs), 3, dtype=torch.float64, device="cuda")
            s.plan = jz.jz_plan_create(s.ctx, s.jobs, s.out, s.est, 0)
        else:
            s.server = jz.jz_server_create(s.ctx, 8 << 30, case["inflight"])
        return s
    n = case["n_traj"]
    s.jobs = [jz.make_params(case["d"], case["L"], case["L_t"], case["beta"],
                             case["l0"] + i * case["l_step"], case["n_step"], case["n_sweep"], n,
                             seed, n_therm=case["n_therm"], direction=case["direction"],
                             update=case["update"], therm_update=case["therm_update"],
                             n_replica=case["n_replica"], whole=case["whole"],
                             protocol=case["protocol"]) for i in range(case["n_l"])]
    where = dict(pin_memory=True) if case["host"] else dict(device="cuda")
    s.out = torch.empty(case["n_l"], n, dtype=torch.int64, **where)
    if case["kind"] == "segment":
        V = case["n_replica"] * case["L_t"] * case["L"] ** (case["d"] - 1)
        s.spins = torch.empty(n, V, dtype=torch.int8, device="cuda")
    return s


# -------------------------------------------------------------------- run --
def _estimates(s):
    """The estimate of every transformation, as (ln <e^-W>, Delta S, its error)."""
    return np.array([jz.estimator_reduce(s.ctx, s.out[i], p.n_traj, p.beta, p.n_step, p.direction)
                     for i, p in enumerate(s.jobs)])


def run(s):
    c = s.case
    if s.kind == "reduce":
        return np.array(jz.estimator_reduce(s.ctx, s.work, c["n"], c["beta"], c["n_step"],
                                            c["direction"], c["bins"]))
    if s.kind == "plan":
        jz.jz_plan_launch(s.plan)
        jz.ising_sync(s.ctx)
        return {"work": torch.cat(s.out), "estimates": s.est}
    if s.kind == "serve":
        ids = [jz.jz_submit(s.server, p) for p in s.jobs]
        est, works = [], []
        for i, p in zip(ids, s.jobs):
            r = jz.jz_wait(s.server, i)
            if r.status != jz.ISING_OK:
                raise jz.IsingError(r.status, "served job")
            w = np.empty(p.n_traj, dtype=np.int64)
            jz.jz_server_work(s.server, i, w)
            works.append(w)
            est.append((r.log_ratio, r.delta_S2, r.delta_S2_err))
        return {"work": np.concatenate(works), "estimates": np.array(est)}
    if s.kind == "segment":
        p, half = s.jobs[0], c["n_step"] // 2
        if half:
            jz.jarzynski_run_segment(s.ctx, p, 0, half, s.out, s.spins)
        jz.jarzynski_run_segment(s.ctx, p, half, c["n_step"], s.out, s.spins)
        return {"work": s.out, "estimates": _estimates(s), "spins": s.spins}
    jz.jarzynski_run_batch(s.ctx, s.jobs, [s.out[i] for i in range(len(s.jobs))])
    return {"work": s.out, "estimates": _estimates(s)}


# ------------------------------------------------------------------ exact --
def exact(case, seed):
    """The estimator in numpy.  A trajectory's whole-number work and its final
    spins have no value in floating point, and an estimate from them none
    without them."""
    if case["kind"] != "reduce":
        return None
    w = _work_values(case, seed).numpy().astype(np.float64)
    x = (-(case["beta"] / case["n_step"]) * w).astype(np.longdouble)
    sign = np.longdouble(-1 if case["direction"] > 0 else 1)

    def log_mean(v):
        m = v.max()
        return m + np.log(np.exp(v - m).sum()) - np.log(np.longdouble(v.size))

    full = log_mean(x)
    n, bins = case["n"], min(case["bins"], case["n"])
    err = np.longdouble(0)
    if bins >= 2:
        edge = [b * (n // bins) for b in range(bins)] + [n]
        theta = np.array([sign * log_mean(np.concatenate([x[:a], x[b:]]))
                          for a, b in zip(edge, edge[1:])])
        err = np.sqrt((bins - 1) * ((theta - theta.mean()) ** 2).sum() / bins)
    return np.array([full, sign * full, err], dtype=np.float64)
