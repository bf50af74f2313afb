"""The work that programs have this framework do, as cases whose passes can be timed.

Every case is a simulation of the extensible bead-spring chain of arXiv:1411.3487 through the public
calls (`Batch`, `Server`), at sizes of this repository's own workloads, experiments and tests:

  steps     a batch that is already running: `step(n)`, then the state is read (`SFP_OBS_MODES_F32`,
            or the FP64 modes of an FP64 batch).  One length, or lengths mixed in one batch.
  sampled   the same with the paper's observables accumulated every few steps on the way.
  start     the equilibrium start that every run begins with, and the conformations it gives.
  serve     jobs of mixed lengths and step counts submitted to a `Server`, waited for and fetched.

Arrays whose values come from an FP32 state are returned as FP32; those of an FP64 batch as FP64.
`exact` is the method written out in torch in 64 bits: tables, noise, force, update and start.
"""
import math

import numpy as np
import torch

import paper_1411_3487_gb300 as sfp
from paper_1411_3487_gb300 import _lib

PRECISION = {"fp32": sfp.SFP_FP32, "bf16": sfp.SFP_MIXED_BF16, "simt": sfp.SFP_FP32_SIMT, "fp64": sfp.SFP_FP64}
LENGTHS = (64, 128, 256, 512)
# steps of the paper's Table 1 in scaled time (1.59, 7.96, 15.9, 15.9 ps)
DTAU = {64: 10.0, 128: 50.0, 256: 100.0, 512: 100.0}


def dtau_of(m):
    """The step of the longest tabulated length that is not above m."""
    return DTAU[max((x for x in LENGTHS if x <= m), default=64)]


def listed():
    return [
        # one dsDNA chain of 64 bp in full precision: the paper's own single-chain runs
        {"name": "one chain 64 fp64", "kind": "steps", "beads": 64, "chains": 1, "precision": "fp64", "steps": 1000},
        # a few sheared chains and a short call: the smallest pool a tumbling study or an interactive loop steps
        {"name": "small 128 shear bf16", "kind": "steps", "beads": 128, "chains": 50, "precision": "bf16",
         "steps": 8, "shear": 1.0e8},
        # the main workload: 4096 chains of 256 bp, mixed precision
        {"name": "main 256 bf16", "kind": "steps", "beads": 256, "chains": 4096, "precision": "bf16", "steps": 400},
        # the same batch in the default precision
        {"name": "main 256 fp32", "kind": "steps", "beads": 256, "chains": 4096, "precision": "fp32", "steps": 300},
        # the long-chain production run: 16384 chains of 512 bp, mixed precision
        {"name": "large 512 bf16", "kind": "steps", "beads": 512, "chains": 16384, "precision": "bf16", "steps": 128},
        # 8192 chains with lengths drawn from the four, each at its own step, from a captured graph
        {"name": "mixed lengths bf16", "kind": "steps", "beads": 0, "chains": 8192, "precision": "bf16",
         "steps": 200, "graph": True},
        # a length that is none of the four, in the default precision: 100 bp, an odd number of chains
        {"name": "odd 100 fp32", "kind": "steps", "beads": 100, "chains": 2001, "precision": "fp32", "steps": 50},
        # the plain FP32 path, which others are checked against
        {"name": "plain 256 fp32", "kind": "steps", "beads": 256, "chains": 1024, "precision": "simt", "steps": 40},
        # a reference ensemble in full precision
        {"name": "ensemble 128 fp64", "kind": "steps", "beads": 128, "chains": 512, "precision": "fp64", "steps": 20},
        # equilibrium runs of the paper's Sec. 5B: observables sampled every 20 steps
        {"name": "sampled 64 bf16", "kind": "sampled", "beads": 64, "chains": 4096, "precision": "bf16",
         "steps": 400, "every": 20},
        # the start of a run
        {"name": "start 256 bf16", "kind": "start", "beads": 256, "chains": 4096, "precision": "bf16"},
        # serving: 120 jobs of the four lengths, half of them sheared, 100 to 2000 steps each
        {"name": "serve bf16", "kind": "serve", "jobs": 120, "low": 100, "high": 2000, "precision": "bf16"},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case.  Steps are bounded so that a pass does no more work than the largest listed case."""
    kind = rng.choice(["steps"] * 6 + ["mixed", "odd", "sampled", "start", "serve", "fp64"])
    if kind == "serve":
        low = _log(rng, 20, 400)
        return {"kind": "serve", "jobs": _log(rng, 4, 200), "low": low, "high": low + _log(rng, 50, 1600),
                "precision": rng.choice(["bf16", "bf16", "fp32"])}
    if kind == "start":
        return {"kind": "start", "beads": rng.choice([20, 64, 100, 128, 200, 256, 512]), "chains": _log(rng, 1, 5000),
                "precision": rng.choice(["bf16", "fp32", "fp64"])}
    if kind == "fp64":
        beads = rng.choice([20, 64, 100, 128, 256])
        chains = _log(rng, 1, 600)
        most = max(1, int(2.0e9 / (18.0 * beads * beads * chains)))
        return {"kind": "steps", "beads": beads, "chains": chains, "precision": "fp64", "steps": _log(rng, 1, min(1000, most) + 1),
                "shear": rng.choice([0.0, 0.0, 1.54e8])}
    if kind == "odd":
        beads, chains = rng.randint(5, 400), _log(rng, 1, 4000)
        precision = rng.choice(["fp32", "bf16", "simt"])
    elif kind == "mixed":
        beads, chains, precision = 0, _log(rng, 16, 9000), rng.choice(["bf16", "bf16", "fp32"])
    else:
        beads, chains = rng.choice(LENGTHS), _log(rng, 1, 12000)
        precision = rng.choice(["bf16", "bf16", "bf16", "fp32", "fp32", "simt"])
    m = beads or 280
    rate = 6.0e12 if precision in ("fp32", "simt") or kind == "odd" else 6.0e13
    most = max(1, int(0.02 * rate / (18.0 * m * m * chains)))
    case = {"kind": "steps", "beads": beads, "chains": chains, "precision": precision,
            "steps": _log(rng, 1, max(2, min(400, most)))}
    if kind == "sampled":
        case.update(kind="sampled", every=rng.choice([1, 7, 20, 50]), steps=max(50, case["steps"]))
        case["chains"] = min(chains, 6000)
    else:
        case["shear"] = rng.choice([0.0, 0.0, 1.0e7, 1.54e8])
        if kind == "mixed":
            case["graph"] = rng.choice([False, True])
    return case


def _bead_counts(case):
    """Beads of each chain: one length, or lengths drawn uniformly from the four (the same for every seed)."""
    if case["beads"]:
        return [case["beads"]] * case["chains"]
    return [int(x) for x in np.random.default_rng(1).choice(LENGTHS, size=case["chains"])]


def _jobs(case):
    """The jobs of a serving run; the seed of a run is its server's noise key."""
    rng = np.random.default_rng(1)
    jobs = []
    for i in range(case["jobs"]):
        m = int(rng.choice(LENGTHS))
        n = int(round(math.exp(rng.uniform(math.log(case["low"]), math.log(case["high"])))))
        shear = float(rng.uniform(1e6, 1e8)) if rng.random() < 0.5 else 0.0
        jobs.append({"n_beads": m, "dtau": DTAU[m], "n_steps": n, "shear_rate_per_s": shear, "job_id": i})
    return jobs


def prepare(case, seed):
    precision = PRECISION[case["precision"]]
    if case["kind"] == "serve":
        return {"case": case, "jobs": _jobs(case),
                "server": sfp.Server(seed=seed, precision=precision, slots_per_pool=256, quantum_steps=64)}
    shear = case.get("shear", 0.0)
    chains = [{"n_beads": m, "dtau": dtau_of(m), "shear_rate_per_s": shear} for m in _bead_counts(case)]
    b = sfp.Batch(chains, seed=seed, precision=precision)
    if case["kind"] != "start":
        b.init_equilibrium()
    if case.get("graph"):
        b.set_graph(True)
    return {"case": case, "batch": b}


def _f32(v):
    return v.astype(np.float32)


def run(state):
    case = state["case"]
    if case["kind"] == "serve":
        server = state["server"]
        tickets = [server.submit(j) for j in state["jobs"]]
        server.wait_idle()
        done = server.poll(len(tickets))
        return {"modes": np.concatenate([_f32(server.modes(t)).ravel() for t in tickets]),
                "steps": np.array([r["n_steps"] for r in sorted(done, key=lambda r: r["ticket"])])}
    b = state["batch"]
    modes = _lib.SFP_OBS_MODES if case["precision"] == "fp64" else _lib.SFP_OBS_MODES_F32
    if case["kind"] == "start":
        b.init_equilibrium()
        return _flat(b.observe(modes))
    if case["kind"] == "sampled":
        b.set_sampling(case["every"])
        b.step(case["steps"])
        return {"modes": _flat(b.observe(modes)), "observables": _f32(b.observe(_lib.SFP_OBS_ACCUM)),
                "power": _f32(b.observe(_lib.SFP_OBS_MODE_POWER)), "com_msd": _f32(b.observe(_lib.SFP_OBS_COM_MSD))}
    b.step(case["steps"])
    return {"modes": _flat(b.observe(modes)), "steps": b.observe(_lib.SFP_OBS_STEP)}


def _flat(v):
    """One array also where the chains of a batch have several lengths."""
    return np.concatenate([x.ravel() for x in v]) if isinstance(v, list) else v


def work(case):
    """The dense transforms in the halves that the mirror symmetry of the modes leaves (9 M flops a bead and step),
    the state read and written once, what is handed to the caller written once."""
    if case["kind"] == "serve":
        steps = (case["high"] - case["low"]) / math.log(case["high"] / case["low"])
        beads = case["jobs"] * sum(LENGTHS) / 4
        return {"bytes": 3 * beads * 12, "flops": 9.0 * case["jobs"] * steps * sum(m * m for m in LENGTHS) / 4}
    es = 8 if case["precision"] == "fp64" else 4
    sizes = LENGTHS if not case["beads"] else (case["beads"],)
    per = case["chains"] / len(sizes)
    values = 3.0 * per * sum(sizes)
    if case["kind"] == "start":
        # the state and its copy for the caller; positions to modes is one transform of three axes
        return {"bytes": 2 * es * values, "flops": 3.0 * per * sum(m * m for m in sizes)}
    extra = values * 4 if case["kind"] == "sampled" else 0.0
    return {"bytes": 3 * es * values + extra, "flops": 9.0 * per * case["steps"] * sum(m * m for m in sizes)}


# ---- the method in 64 bits -------------------------------------------------------------------------------------


def _philox(seed, job, step, call, tag):
    """Words of Philox4x32-10 for counters (step, step >> 32, call, tag) and keys (seed, job), int64 tensors."""
    low = 0xFFFFFFFF
    c = [step & low, (step >> 32) & low, call, torch.full_like(call, tag)]
    c = [x.expand(torch.broadcast_shapes(job.shape, step.shape, call.shape)) for x in c]
    k0, k1 = seed, job
    for r in range(10):
        if r:
            k0, k1 = (k0 + 0x9E3779B9) & low, (k1 + 0xBB67AE85) & low
        p0, p1 = c[0] * 0xD2511F53, c[2] * 0xCD9E8D57
        c = [((p1 >> 32) & low) ^ c[1] ^ k0, p1 & low, ((p0 >> 32) & low) ^ c[3] ^ k1, p0 & low]
    return c


def _uniform(x):
    return ((x >> 9).double() + 0.5) * 2.0 ** -23


def _normals(seed, job, step, m):
    """Bead normals [chains][3][m]: normal 3 n + axis of a chain and step is value k mod 4 of Philox call k // 4."""
    calls = (3 * m + 3) // 4
    w = _philox(seed, job[:, None], step[:, None], torch.arange(calls, device=job.device)[None], 0)
    ra, rb = torch.sqrt(-2 * torch.log(_uniform(w[0]))), torch.sqrt(-2 * torch.log(_uniform(w[2])))
    ta, tb = 2 * math.pi * _uniform(w[1]), 2 * math.pi * _uniform(w[3])
    g = torch.stack([ra * torch.cos(ta), ra * torch.sin(ta), rb * torch.cos(tb), rb * torch.sin(tb)], -1)
    return g.reshape(job.shape[0], -1)[:, :3 * m].reshape(-1, m, 3).transpose(1, 2)


class _Exact:
    """Chains of one length in FP64: T* = 0.034, nu = 0.35, a = 0.33 nm, a^2 xi / kT = 52.0 ps."""

    T, NU, A, A2XI = 0.034, 0.35, 0.33, 52.0

    def __init__(self, m, dtau, seed, jobs, shear=None):
        dev = "cuda" if torch.cuda.is_available() else "cpu"
        d = dict(dtype=torch.float64, device=dev)
        self.m, self.dtau, self.seed = m, dtau, int(seed)
        self.job = torch.as_tensor(np.asarray(jobs, dtype=np.int64), device=dev)
        self.c_ps = self.T * (1 - 2 * self.NU) ** 2 * self.A2XI
        rate = torch.zeros(len(jobs), **d) if shear is None else torch.as_tensor(np.asarray(shear, dtype=np.float64), **d)
        self.shear = rate * self.c_ps * 1e-12
        n, p = torch.arange(m, **d)[:, None], torch.arange(m, **d)[None]
        self.phi = math.sqrt(2.0 / m) * torch.cos(math.pi * p * (n + 0.5) / m)
        self.phi[:, 0] = 1 / math.sqrt(m)
        # phi_n - phi_{n-1} = -2 sqrt(2/M) sin(pi p n / M) sin(pi p / 2 M)
        self.chi = -2 * math.sqrt(2.0 / m) * torch.sin(math.pi * (p * n) / m) * torch.sin(math.pi * p / (2 * m))
        self.chi[0], self.chi[:, 0] = 0, 0
        s2 = torch.sin(math.pi * p[0] / (2 * m)) ** 2
        zeta, gap = 16 * self.NU * s2 * s2, (1 - 2 * self.NU) * 4 * s2
        zeta[0], gap[0] = 1, 1
        self.dm = -torch.expm1(-zeta * dtau)
        self.h = torch.exp(-zeta * dtau) * -torch.expm1(-gap * dtau) / gap
        self.w = torch.sqrt(self.T * -torch.expm1(-2 * zeta * dtau) / zeta)
        self.g = self.dm / zeta
        self.dm[0], self.h[0], self.w[0], self.g[0] = 0, 0, math.sqrt(2 * self.T * dtau), dtau
        self.R = torch.zeros(len(jobs), 3, m, **d)
        self.t = torch.zeros(len(jobs), dtype=torch.int64, device=dev)

    def start(self):
        """The equilibrium sampler: bond lengths about the straight rod, von Mises-Fisher tangents, centre at 0."""
        m, n, dev = self.m, self.m - 1, self.R.device
        c, l0, ld, lo = self.job.shape[0], np.zeros(self.m - 1), np.zeros(self.m - 1), np.zeros(self.m - 1)
        band = np.zeros((n, n)) + np.eye(n) - self.NU * (np.eye(n, k=1) + np.eye(n, k=-1))
        l0 = np.linalg.solve(band, np.ones(n))
        ld[0] = 1.0
        for i in range(1, n):
            lo[i] = -self.NU / ld[i - 1]
            ld[i] = math.sqrt(1 - lo[i] * lo[i])
        w = _philox(self.seed, self.job[:, None], torch.zeros(1, 1, dtype=torch.int64, device=dev),
                    torch.arange(m, device=dev)[None], 1)
        u = [_uniform(x) for x in w]
        eps = torch.sqrt(-2 * torch.log(u[0])) * torch.cos(2 * math.pi * u[1])
        x = torch.zeros(c, n, dtype=torch.float64, device=dev)
        for i in range(n - 1, -1, -1):
            x[:, i] = (eps[:, i + 1] - (float(lo[i + 1]) * x[:, i + 1] if i + 1 < n else 0.0)) / float(ld[i])
        length = torch.as_tensor(l0, device=dev) + math.sqrt(self.T) * x
        cos0 = 2 * u[0][:, 0] - 1
        sin0, turn = torch.sqrt((1 - cos0) * (1 + cos0)), 2 * math.pi * u[1][:, 0]
        t = torch.stack([sin0 * torch.cos(turn), sin0 * torch.sin(turn), cos0], 1)
        kappa = self.NU * length[:, :-1] * length[:, 1:] / self.T
        uz, turn = u[2][:, 2:], 2 * math.pi * u[3][:, 2:]
        ct = 1 + torch.log(uz + (1 - uz) * torch.exp(-2 * kappa)) / kappa
        st = torch.sqrt(torch.clamp((1 - ct) * (1 + ct), min=0))
        ca, sa = st * torch.cos(turn), st * torch.sin(turn)
        bonds = [length[:, 0:1] * t]
        for i in range(1, n):
            tx, ty, tz = t.unbind(1)
            sg = torch.copysign(torch.ones_like(tz), tz)
            a = -1 / (sg + tz)
            b = tx * ty * a
            e1 = torch.stack([1 + sg * tx * tx * a, sg * b, -sg * tx], 1)
            e2 = torch.stack([b, sg + ty * ty * a, -ty], 1)
            t = ct[:, i - 1, None] * t + ca[:, i - 1, None] * e1 + sa[:, i - 1, None] * e2
            t = t / t.norm(dim=1, keepdim=True)
            bonds.append(length[:, i:i + 1] * t)
        r = torch.zeros(c, 3, m, dtype=torch.float64, device=dev)
        r[:, :, 1:] = torch.stack(bonds, 2).cumsum(2)
        self.R = (r - r.mean(2, keepdim=True)) @ self.phi
        self.R[:, :, 0] = 0
        self.t.zero_()
        return self

    def step(self, n, stop=None):
        m = self.m
        for _ in range(n):
            u = self.R @ self.chi.T
            inv = torch.rsqrt((u * u).sum(1, keepdim=True))
            inv[:, :, 0] = 0
            force = u * (inv - (1 - 2 * self.NU))
            z = _normals(self.seed, self.job, self.t, m) @ self.phi
            new = self.R - self.dm * self.R + self.h * (force @ self.chi) + self.w * z
            new[:, 0] += self.shear[:, None] * self.g * self.R[:, 1]
            if stop is None:
                self.R, self.t = new, self.t + 1
            else:
                go = self.t < stop
                self.R, self.t = torch.where(go[:, None, None], new, self.R), self.t + go.long()
        return self

    def sample(self, acc):
        """Adds one sample: |L|^2, |u_m|^2, |r_m - r_cm|^2 (nm^2), mode powers, centre-of-mass windows."""
        m, d2 = self.m, (self.A * (1 - 2 * self.NU)) ** 2
        mid = (m - 1) // 2
        ends = (self.R * (self.phi[m - 1] - self.phi[0])).sum(2)
        bond = (self.R * self.chi[m // 2]).sum(2)
        bead = (self.R[:, :, 1:] * self.phi[mid, 1:]).sum(2)
        one = torch.ones_like(ends[:, 0])
        acc["observables"] = acc.get("observables", 0) + torch.stack(
            [(ends ** 2).sum(1) * d2, (bond ** 2).sum(1) * d2, (bead ** 2).sum(1) * d2, one], 1)
        acc["power"] = acc.get("power", 0) + self.R ** 2
        k, com = acc.get("k", 0), self.R[:, :, 0] / math.sqrt(m)
        msd, snap = acc.setdefault("com_msd", torch.zeros(len(com), 4, 2, dtype=com.dtype, device=com.device)), acc.setdefault("snap", {})
        for i, lag in enumerate((1, 10, 100, 1000)):
            if k % lag == 0:
                if k:
                    msd[:, i, 0] += ((com - snap[i]) ** 2).sum(1) * d2
                    msd[:, i, 1] += 1
                snap[i] = com.clone()
        acc["k"] = k + 1


def exact(case, seed):
    if case["kind"] == "serve":
        jobs = _jobs(case)
        out = [None] * len(jobs)
        for m in LENGTHS:
            at = [i for i, j in enumerate(jobs) if j["n_beads"] == m]
            if not at:
                continue
            n = [jobs[i]["n_steps"] for i in at]
            e = _Exact(m, DTAU[m], seed, at, [jobs[i]["shear_rate_per_s"] for i in at]).start()
            e.step(max(n), torch.as_tensor(n, device=e.R.device))
            for k, i in enumerate(at):
                out[i] = e.R[k].cpu().numpy().ravel()
        return {"modes": np.concatenate(out), "steps": np.array([j["n_steps"] for j in jobs])}
    beads = np.array(_bead_counts(case))
    if case["kind"] != "start" and float((beads.astype(float) ** 2).sum()) * 18 * case["steps"] > 1.2e13:
        return None
    rows = [None] * len(beads)
    steps = np.full(len(beads), case.get("steps", 0), dtype=np.int64)
    for m in sorted(set(beads.tolist())):
        at = np.flatnonzero(beads == m)
        e = _Exact(m, dtau_of(m), seed, at, np.full(len(at), case.get("shear", 0.0))).start()
        if case["kind"] == "sampled":
            acc, left = {}, case["steps"]
            e.sample(acc)
            while left >= case["every"]:
                e.step(case["every"]).sample(acc)
                left -= case["every"]
            e.step(left)
            return {"modes": e.R.cpu().numpy(), "observables": acc["observables"].cpu().numpy(),
                    "power": acc["power"].cpu().numpy(), "com_msd": acc["com_msd"].cpu().numpy()}
        if case["kind"] == "steps":
            e.step(case["steps"])
        if len(at) == len(beads):
            return e.R.cpu().numpy() if case["kind"] == "start" else {"modes": e.R.cpu().numpy(), "steps": steps}
        for k, i in enumerate(at):
            rows[i] = e.R[k].cpu().numpy().ravel()
    return {"modes": np.concatenate(rows), "steps": steps}
