"""Workloads of the library through its public entry points, for timing.

Each case is what a program that uses the library does in earnest: a served
request from its configuration to its diagnostics, a long-lived run advanced
between two readings of its diagnostics, a batch of resident runs advanced by
one RF period, a sweep, and the kernel-level deposit.  The sizes are those of
the recipes in ``paper_2308_13092_gb300/inputs.py`` and of the paper's Table 1.
"""
from __future__ import annotations

import math

import numpy as np
import torch

QE, ME, AMU, KB, EPS0 = 1.602176634e-19, 9.1093837015e-31, 1.66053906660e-27, 1.380649e-23, 8.8541878128e-12

# schemes of the library: EC, MC (linear deposit), EC2, MC2 (quadratic deposit)
EC, MC, EC2, MC2 = 0, 1, 2, 3


# ------------------------------------------------------------------ the cases
def _request(name, cells, per_species, steps, **kw):
    c = dict(kind="request", cells=cells, per_species=per_species, steps=steps, sample_every=steps // 10,
             grid="uniform", scheme=EC, density=1.288e15, steps_per_period=750, volts=300.0, mtorr=30.0)
    c.update(kw)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # One RF period of the smallest discharge anyone studies (128 cells, 64
        # particles per cell and species): launches and latency count.
        _request("small_request", 128, 8192, 200, density=5e13, steps_per_period=200, sample_every=20),
        # The ordinary single run: 1024 cells at the Debye length, 524,288 particles.
        _request("resolved_request", 1024, 262144, 150),
        # The same plasma at twice the cell size with the momentum-conserving
        # scheme that the energy-conserving one is compared with.
        _request("mc_request", 512, 131072, 150, scheme=MC),
        # A non-uniform doubling grid (114 cells, odd particle count), the
        # paper's way of using fewer cells.
        _request("doubling_request", 114, 29127, 150, grid="doubling", dx_min=4, dx_max=32),
        # The paper's own discharge: 2048 cells, 512 particles per cell, 1000 V;
        # the smallest time step, so few collision candidates.
        _request("paper_request", 2048, 1048576, 100, density=7e15, steps_per_period=4000, volts=1000.0),
        # A long-lived run with particle rebalancing on the doubling grid
        # (weight multipliers, merges and splits every 20 steps).
        dict(name="rebalanced_run", kind="rebalanced", cells=114, per_species=29127, steps=100, sample_every=10,
             grid="doubling", dx_min=4, dx_max=32, scheme=EC, density=1.288e15, steps_per_period=750,
             volts=300.0, mtorr=30.0, every=20, target=256, lo=128, hi=384, m0=16),
        # A long-lived collisionless plasma with the higher-order scheme,
        # electrons and mobile ions, its particles read as a checkpoint.
        dict(name="higher_order_run", kind="periodic", runs=1, cells=1024, ppc=64, ions=True, scheme=EC2, other=EC2,
             dx_lambda=4.0, dt_wpe=0.1, density=1e14, te=2.0, quiet=False, steps=200, sample_every=20),
        # The heating sweep of the paper's Appendix B as one batch: both
        # schemes at six resolutions, 2048 cells, 64 particles per cell.
        dict(name="heating_sweep", kind="sweep", runs=12, cells=2048, ppc=64, ions=False, scheme=EC, other=MC,
             dx_lambda=0.5, dt_wpe=0.1, density=7e15, te=2.585, quiet=True, steps=200, sample_every=100),
        # A wave of 64 served requests from submission to their diagnostics.
        dict(name="served_wave", kind="wave", runs=64, sizes=8, scale=1.0, steps=200, sample_every=40),
        # The main workload: 256 resident runs of 1e4 to 1e6 particles (5e7 in
        # all) advanced by one RF period, then every run's diagnostics.
        dict(name="resident_batch", kind="batch", runs=256, sizes=0, scale=1.0, steps=400, sample_every=40),
        # The kernel-level charge deposit on caller-owned arrays, in cell order
        # up to one step's drift.
        dict(name="deposit", kind="deposit", cells=1024, n=16777259, order=1, bc=0, noalloc=False, ordered=True),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["request"] * 4 + ["rebalanced", "periodic", "wave", "batch", "deposit"])
    if kind in ("request", "rebalanced"):
        dense = rng.random() < 0.6
        c = _request(None, int(_log(rng, 64, 2048)), int(_log(rng, 4096, 1.05e6)), 0,
                     density=_log(rng, 3e14, 1.5e15) if dense else _log(rng, 5e13, 3e14),
                     steps_per_period=750 if dense else 400, volts=_log(rng, 100, 500), mtorr=_log(rng, 10, 100),
                     scheme=rng.choice([EC, EC, EC, MC, EC2, MC2]))
        c["steps"] = max(20, min(int(_log(rng, 60, 400)), int(2e8 / c["per_species"])))
        c["sample_every"] = max(1, c["steps"] // rng.randint(2, 12))
        if kind == "rebalanced" or (c["scheme"] < EC2 and rng.random() < 0.4):
            c["scheme"] = min(c["scheme"], MC)
            c["grid"] = "tanh" if rng.random() < 0.4 else "doubling"
            if c["grid"] == "doubling":
                c["dx_min"], c["dx_max"] = rng.choice([(1, 8), (2, 16), (4, 32)])
                c["cells"] = _doubling_edges(c["dx_min"], c["dx_max"]).size - 1
            else:
                c["cells"] = rng.randint(100, 400)
            c["per_species"] = min(c["per_species"], 200000)
        if kind == "rebalanced":
            target = max(8, min(1024, c["per_species"] // c["cells"]))
            c.update(kind=kind, every=rng.choice([10, 20, 50]), target=target, lo=target // 2,
                     hi=target + target // 2, m0=16)
        return c
    if kind == "periodic":
        s = rng.choice([EC, MC, EC2, MC2])
        return dict(kind=kind, runs=1, cells=int(_log(rng, 64, 2048)), ppc=rng.randint(16, 256), ions=rng.random() < 0.5,
                    scheme=s, other=s, dx_lambda=_log(rng, 1.0, 8.0), dt_wpe=0.1, density=1e14, te=2.0,
                    quiet=rng.random() < 0.3, steps=rng.randint(20, 80), sample_every=20)
    if kind == "wave":
        return dict(kind=kind, runs=rng.randint(8, 100), sizes=rng.randint(1, 1000), scale=1.0,
                    steps=rng.randint(60, 300), sample_every=rng.choice([20, 40]))
    if kind == "batch":
        return dict(kind=kind, runs=int(_log(rng, 8, 256)), sizes=rng.randint(1, 1000), scale=_log(rng, 0.1, 1.0),
                    steps=rng.randint(100, 300), sample_every=rng.choice([20, 40]))
    noalloc = rng.random() < 0.4
    return dict(kind="deposit", cells=int(_log(rng, 16, 2048)), n=int(_log(rng, 1e4, 6e7)),
                order=1 if noalloc else rng.choice([1, 1, 2]), bc=rng.choice([0, 1]), noalloc=noalloc,
                ordered=rng.random() < 0.7)


# ------------------------------------------------------------------ the inputs
def _doubling_edges(dx_min, dx_max):
    from paper_2308_13092_gb300 import ecpic
    return ecpic.ecpic_doubling_grid(1024, 0.3, 0.05, dx_min, dx_max)


def _discharge(case, seed):
    """A discharge's configuration, as a program of the library writes it."""
    from paper_2308_13092_gb300 import inputs as I
    edges = None
    if case["grid"] == "doubling":
        edges = _doubling_edges(case["dx_min"], case["dx_max"])
    elif case["grid"] == "tanh":
        edges = I.tanh_edges(case["cells"], I.L_GAP, 0.4 * I.L_GAP / case["cells"])
    c = I.ccp("run", N=case["cells"], n0=case["density"], dt=1.0 / (case["steps_per_period"] * I.F_RF), ppc=0,
              v0=case["volts"], p_mtorr=case["mtorr"], n_steps=case["steps"], seed=seed, scheme=case["scheme"],
              edges=edges, n_per_species=case["per_species"])
    c.sample_every = case["sample_every"]
    if case["kind"] == "rebalanced":
        c.rebalance = {k: case[k] for k in ("every", "target", "lo", "hi", "m0")}
    return c


def _periodic(case, seed):
    """The configurations of a collisionless periodic case: for a sweep, both
    schemes at runs/2 resolutions, each twice the one before."""
    from paper_2308_13092_gb300 import inputs as I
    out = []
    for r in range(case["runs"]):
        scheme, dx = _periodic_run(case, r)
        c = I.periodic_plasma(N=case["cells"], dx_lambda=dx, ppc=case["ppc"], dt_wpe=case["dt_wpe"],
                              n_steps=case["steps"], seed=1000 * seed + r, scheme=scheme, ions=case["ions"],
                              n0=case["density"], Te=case["te"], quiet=case["quiet"])
        c.sample_every = case["sample_every"]
        out.append(c)
    return out


def _periodic_run(case, r):
    half = max(1, case["runs"] // 2)
    return (case["scheme"] if r < half else case["other"]), case["dx_lambda"] * 2.0 ** (r % half)


def _manifest(case, seed):
    from paper_2308_13092_gb300 import inputs as I
    runs = I.batched_manifest(case["runs"], seed=case["sizes"], scale=case["scale"],
                              steps=4400 if case["kind"] == "batch" else case["steps"])
    for r, c in enumerate(runs):
        c.seed = 1000003 * seed + r
        c.sample_every = case["sample_every"]
    return runs


def prepare(case, seed):
    from paper_2308_13092_gb300 import ecpic
    kind = case["kind"]
    st = dict(kind=kind, steps=case.get("steps", 0))
    if kind == "deposit":
        g = torch.Generator(device="cuda").manual_seed(seed)
        N, n = case["cells"], case["n"]
        cell = torch.randint(0, N, (n,), generator=g, device="cuda", dtype=torch.int32)
        if case["ordered"]:  # sorted, then drifted by up to a cell, a few absorbed
            cell = torch.sort(cell).values
            cell += torch.randint(-1, 2, (n,), generator=g, device="cuda", dtype=torch.int32)
            cell[cell >= N] = -1
        st.update(case=dict(case), cell=cell, xi=torch.rand(n, generator=g, device="cuda"),
                  S=torch.zeros(N + 1, dtype=torch.int64, device="cuda"))
    elif kind == "request":
        st["config"] = _discharge(case, seed)
        st["engine"] = ecpic.Engine(max_slots=1, max_cells=st["config"].N, species_per_run=2)
    elif kind == "rebalanced":
        st["run"] = ecpic.Run.from_config(_discharge(case, seed))
        st["run"].set_auto_grow(True)
    elif kind == "periodic":
        st["run"] = ecpic.Run.from_config(_periodic(case, seed)[0])
    elif kind == "sweep":
        st["configs"] = _periodic(case, seed)
        st["engine"] = ecpic.Engine(max_slots=case["runs"], max_cells=case["cells"],
                                    species_per_run=2 if case["ions"] else 1)
    else:
        st["configs"] = _manifest(case, seed)
        st["engine"] = ecpic.Engine(max_slots=case["runs"], max_cells=1024, species_per_run=2)
        if kind == "batch":  # resident for good: a pass advances them
            st["tickets"] = [st["engine"].submit(c, 1 << 40) for c in st["configs"]]
            st["engine"].pump(0)
    return st


# ------------------------------------------------------------------ a pass
def _counts(d):
    return np.array([[s["n"], s["absorbed_left"], s["absorbed_right"], s["births"], s["lost"], s["candidates"],
                      s["clamps"], s["impacts_dropped"], s["rb_merged"], s["rb_split"], s["rb_skipped"]]
                     + s["collisions"] for s in d["species"]], dtype=np.int64)


def _by_id(p):
    """Particles of a run without births or losses: row i is particle i."""
    out = {k: np.empty_like(p[k]) for k in ("cell", "xi", "vx", "vy", "vz")}
    for k, v in out.items():
        v[p["id"]] = p[k]
    return out


def _outputs(diags):
    """What the diagnostics of the runs hold, run after run in one array each."""
    out = {k: np.concatenate([d[k].ravel() for d in diags])
           for k in ("density", "phi", "Tx", "Tx_mom", "power", "eedf", "iedf", "iad", "ke")}
    out["fe"] = np.array([d["fe"] for d in diags])
    out["levels"] = np.array([[d["step"], d["n_samples"]] for d in diags], dtype=np.int64)
    out["counts"] = np.concatenate([_counts(d) for d in diags])
    return out


def run(state):
    kind = state["kind"]
    if kind == "deposit":
        return _deposit(state)
    if kind in ("rebalanced", "periodic"):
        r = state["run"]
        r.step(state["steps"])
        r.sync()
        out = _outputs([r.diagnostics()])
        out["field"] = r.fields()
        if kind == "periodic":
            out["particles"] = [_by_id(r.get_particles(s)) for s in range(r.ns)]
        return out
    eng = state["engine"]
    if kind == "batch":
        eng.pump(state["steps"])
        return _outputs([eng.poll(t, diagnostics=True, profiles=True)["diag"] for t in state["tickets"]])
    configs = [state["config"]] if kind == "request" else state["configs"]
    tickets = [eng.submit(c) for c in configs]
    resident, queued = eng.pump(state["steps"])
    while resident or queued:
        resident, queued = eng.pump(state["steps"])
    diags = [eng.poll(t, diagnostics=True, profiles=True)["diag"] for t in tickets]
    for t in tickets:
        eng.release(t)
    return _outputs(diags)


def _deposit(state):
    from paper_2308_13092_gb300 import ecpic
    c, S = state["case"], state["S"]
    S.zero_()
    args = (c["n"], state["cell"].data_ptr(), state["xi"].data_ptr(), S.data_ptr(),
            torch.cuda.current_stream().cuda_stream or None)
    if c["order"] == 2:
        ecpic.ecpic_deposit_device2(c["cells"], c["bc"], *args)
    elif c["noalloc"]:
        ecpic.ecpic_deposit_device_noalloc(c["cells"], *args)
    else:
        ecpic.ecpic_deposit_device(c["cells"], *args)
    return S


# ------------------------------------------------------------------ the work
def work(case):
    """Bytes of the particle records that a step cannot do without (cell, offset
    and x velocity read and written: 24 B; the id for a collision draw: 8 B; the
    other two velocities for an electron's collision test: 8 B; the weight
    multiplier: 4 B) and its floating-point operations; the load of a run that
    starts in the pass (28 B)."""
    kind = case["kind"]
    if kind == "deposit":
        return {"bytes": 8 * case["n"] + 8 * (case["cells"] + 1), "flops": 4 * case["n"]}
    if kind in ("periodic", "sweep"):
        n = case["runs"] * case["cells"] * case["ppc"] * (2 if case["ions"] else 1)
        start = 28 * n if kind == "sweep" else 0
        return {"bytes": 24 * n * case["steps"] + start, "flops": 15 * n * case["steps"]}
    if kind in ("request", "rebalanced"):
        n = 2 * case["per_species"]
    else:
        rng = np.random.default_rng(case["sizes"])
        n = 0
        for _ in range(case["runs"]):  # the draws of the manifest, in its order
            rng.uniform(math.log(64), math.log(1024))
            n += 2 * max(int(round(np.exp(rng.uniform(math.log(1e4), math.log(1e6))) * case["scale"])) // 2, 16)
            rng.uniform(0, 1, 3)
    per = 36 + (4 if kind == "rebalanced" else 0)  # electrons 40, ions 32
    start = 28 * n if kind in ("request", "wave") else 0
    return {"bytes": per * n * case["steps"] + start, "flops": 25 * n * case["steps"]}


# ------------------------------------------------------------------ in 64 bits
def exact(case, seed):
    """The collisionless cases in 64-bit floats and the deposit in 64-bit
    integers, in plain torch.  A discharge with collisions has no such value: a
    collision is taken or not by comparing a random number with a rate, so a
    last bit of a velocity sends its trajectory another way."""
    if case["kind"] == "deposit":
        return _exact_deposit(case, seed)
    if case["kind"] not in ("periodic", "sweep"):
        return None
    runs = [_exact_periodic(case, 1000 * seed + r, *_periodic_run(case, r)) for r in range(case["runs"])]
    out = {k: np.concatenate([r[k].ravel() for r in runs])
           for k in ("density", "phi", "Tx", "Tx_mom", "power", "ke", "fe")}
    out.update(eedf=None, iedf=None, iad=None, levels=None, counts=None)
    if case["kind"] == "periodic":
        out["field"] = {"phi": runs[0]["field_phi"], "E": runs[0]["field_E"]}
        out["particles"] = [dict(cell=None, xi=None, vx=p[1].cpu().numpy(), vy=p[2].cpu().numpy(), vz=p[3].cpu().numpy())
                            for p in runs[0]["particles"]]
    return out


def _exact_deposit(case, seed):
    st = prepare(case, seed)
    N, periodic = case["cells"], case["bc"] == 1
    S = torch.zeros(N + 1, dtype=torch.int64, device="cuda")
    ok = st["cell"] >= 0
    c = st["cell"][ok].long()
    r = torch.floor(st["xi"][ok].double() * 2.0 ** 32).long()
    if case["order"] == 1:
        S.index_add_(0, c, 2 ** 32 - r)
        S.index_add_(0, c + 1, r)
        return S
    up = (r >= 2 ** 31).long()
    n0, u = c + up, r - (up << 32)
    a = _half_square(2 ** 31 - u)
    b = _half_square(2 ** 31 + u)
    for node, share in ((n0 - 1, a), (n0, 2 ** 32 - a - b), (n0 + 1, b)):
        S.index_add_(0, node % N if periodic else node.clamp(0, N), share)
    if periodic:
        S[N] = S[0]
    return S


def _half_square(v):
    """floor(v^2 / 2^33) for 0 <= v <= 2^32, in signed 64-bit integers."""
    hi, lo = v >> 17, v & (2 ** 17 - 1)  # v^2 = hi^2 2^34 + hi lo 2^18 + lo^2
    return (hi * hi << 1) + ((hi * lo * 2 + ((lo * lo) >> 17)) >> 16)


def _philox(i, word3, seed):
    m32 = 0xFFFFFFFF
    c = [i & m32, i >> 32, torch.full_like(i, m32), torch.full_like(i, word3)]
    k0, k1 = seed & m32, seed >> 32
    for _ in range(10):
        p0, p1 = c[0] * 0xD2511F53, c[2] * 0xCD9E8D57
        c = [((p1 >> 32) & m32) ^ c[1] ^ k0, p1 & m32, ((p0 >> 32) & m32) ^ c[3] ^ k1, p0 & m32]
        k0, k1 = (k0 + 0x9E3779B9) & m32, (k1 + 0xBB67AE85) & m32
    return c


def _exact_periodic(case, seed, scheme, dx_lambda):
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    f64 = dict(dtype=torch.float64, device=dev)
    N, te, n0 = case["cells"], case["te"], case["density"]
    lam = math.sqrt(EPS0 * te / (n0 * QE))
    dt = case["dt_wpe"] / math.sqrt(n0 * QE * QE / (EPS0 * ME))
    L = N * dx_lambda * lam
    dx, n = L / N, N * case["ppc"]
    w = n0 * L / n
    species = [(-QE, ME, te)] + ([(QE, 4 * AMU, 0.5)] if case["ions"] else [])
    ns = len(species)
    part = []
    for s, (q, m, T) in enumerate(species):
        i = torch.arange(n, dtype=torch.int64, device=dev)
        A, B = _philox(i, (s << 8) | 0x80, seed), _philox(i, (s << 8) | 0x81, seed)
        X = (i.double() + 0.5) / n if case["quiet"] else A[0].double() / 2.0 ** 32
        u = [b.double() / 2.0 ** 32 for b in B]
        ra, rb = (torch.sqrt(-2 * torch.log(v + 2.0 ** -32)) for v in (u[0], u[2]))
        sd = math.sqrt(QE * T / m)
        part.append([X * N, sd * ra * torch.cos(2 * math.pi * u[1]), sd * ra * torch.sin(2 * math.pi * u[1]),
                     sd * rb * torch.cos(2 * math.pi * u[3])])

    def nodes(x, order):
        """Nodes (mod N) and shares of positions x in cells."""
        if order == 1:
            c = torch.floor(x).long()
            t = x - c
            return [(c % N, 1 - t), ((c + 1) % N, t)]
        c = torch.floor(x + 0.5).long()
        u = x - c
        return [((c - 1) % N, 0.5 * (0.5 - u) ** 2), (c % N, 0.75 - u * u), ((c + 1) % N, 0.5 * (0.5 + u) ** 2)]

    def add(x, order, values=None):
        S = torch.zeros(N, **f64)
        for node, share in nodes(x, order):
            S.index_add_(0, node, share if values is None else share * values)
        return S

    order = 2 if scheme >= EC2 else 1

    def solve():
        S = [add(p[0], order) for p in part]
        Q = sum(q * w * s for (q, _, _), s in zip(species, S))
        C = torch.zeros(N, **f64)
        C[1:] = torch.cumsum(Q - Q.sum() / N, 0)[1:] - (Q - Q.sum() / N)[0]
        g = (C.sum() * dx / EPS0) / L - C / EPS0
        phi = torch.zeros(N + 1, **f64)
        phi[1:] = torch.cumsum(g * dx, 0)
        phi[N] = 0.0
        return S, g, phi

    S, g, phi = solve()
    acc = {k: [torch.zeros(N, **f64) for _ in range(ns)] for k in ("D", "T", "M1", "M2", "P")}
    acc_phi, samples = torch.zeros(N + 1, **f64), 0
    ke, fe = np.zeros(ns), 0.0
    for k in range(case["steps"]):
        sample = (k + 1) % case["sample_every"] == 0
        face = -g
        node = -0.5 * (g + torch.roll(g, 1))
        if sample:
            fe = float(0.5 * EPS0 * (g * g).sum() * dx)
            samples += 1
        for s, (q, m, _) in enumerate(species):
            x, v = part[s][0], part[s][1]
            if scheme == EC:
                E = face[torch.floor(x).long() % N]
            elif scheme == EC2:
                c = torch.floor(x + 0.5).long()
                E = (0.5 - (x - c)) * face[(c - 1) % N] + (0.5 + (x - c)) * face[c % N]
            else:
                E = sum(t * node[i] for i, t in nodes(x, order))
            vn = v + q / m * dt * E
            if sample:
                acc["P"][s].index_add_(0, torch.floor(x).long() % N, (v + vn) * E)
                ke[s] = float(0.5 * m * w * (v * vn + part[s][2] ** 2 + part[s][3] ** 2).sum())
            part[s][0], part[s][1] = torch.remainder(x + vn * dt / dx, N), vn
        S, g, phi = solve()
        if sample:
            acc_phi += phi
            for s, (q, m, _) in enumerate(species):
                M1, M2 = (add(part[s][0], 1, part[s][1] ** p) for p in (1, 2))
                D = S[s]
                one = torch.where(D > 0, D, torch.ones_like(D))
                acc["T"][s] += torch.where(D > 0, m / QE * (M2 / one - (M1 / one) ** 2), torch.zeros_like(D))
                for key, v in (("D", D), ("M1", M1), ("M2", M2)):
                    acc[key][s] += v

    def ends(v):
        return torch.cat([v, v[:1]]).cpu().numpy()

    inv = 1.0 / samples if samples else 0.0
    mom = [torch.where(d > 0, m / QE * (b / d.clamp(min=1e-300) - (a / d.clamp(min=1e-300)) ** 2), torch.zeros_like(d))
           for (q, m, _), d, a, b in zip(species, acc["D"], acc["M1"], acc["M2"])]
    return dict(particles=part, density=np.stack([w * ends(d) * inv / dx for d in acc["D"]]), phi=acc_phi.cpu().numpy() * inv,
                Tx=np.stack([ends(t) * inv for t in acc["T"]]), Tx_mom=np.stack([ends(t) for t in mom]),
                power=np.stack([0.5 * q * w * p.cpu().numpy() / dx * inv for (q, _, _), p in zip(species, acc["P"])]),
                ke=ke, fe=np.array([fe]), field_phi=phi.cpu().numpy(),
                field_E=(-g).cpu().numpy() if scheme in (EC, EC2) else ends(-0.5 * (g + torch.roll(g, 1))))
