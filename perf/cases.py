"""Workloads of the library in use: Monte Carlo sweeps of projective determinant-QMC chains, and the Green's function of given fields.

A program holds a context (its model, trial state and Markov chains live on the GPU) and calls ``sweep`` once per pass, then reads the
records of every chain in one copy: that is one pass of a ``sweep`` case.  Programs that follow a few chains closely also read their G
and fields, so contexts of at most four chains return those too.  A ``green`` case is the other use: fields made elsewhere go in, the
equal-time Green's functions and the weight come out.

Values that the reduced-precision paths hold in FP32 (G, and the estimates taken from it) are returned as FP32; the FP64 path's as FP64.
"""
import math

import numpy as np

from paper_2303_13403_gb300 import pqmc, workloads

PRECISION = {"fp64": pqmc.FP64, "fp32": pqmc.FP32, "bf16x3": pqmc.BF16X3}
FEW = 4                 # contexts of at most this many chains return G and the fields as well
MAX_SECONDS = 0.2       # what a drawn case may cost at most, by estimate()


def _case(model, Lx, Ly, prec, chains, two_theta, **kw):
    c = {"use": "sweep", "model": model, "Lx": Lx, "Ly": Ly, "prec": prec, "chains": chains, "two_theta": two_theta,
         "n_stab": 10 if prec == "fp64" else 2, "U": 4.0, "g": 0.6, "M_N": 0.21, "spread": False}
    c.update(kw)
    return c


def listed():
    out = []

    def add(name, *a, **kw):
        out.append(dict(_case(*a, **kw), name=name))

    # one small plain chain in FP64: the reference run of a new model, and the check of a new machine; one CTA, all latency
    add("plain18-fp64-1", "honeycomb", 3, 3, "fp64", 1, 10.0, g=0.0, M_N=0.0)
    # one Gutzwiller chain of 72 sites: a user looks at one trajectory
    add("gutz72-fp32-1", "honeycomb", 6, 6, "fp32", 1, 8.0)
    # the benchmark's production batch: 608 chains of 72 sites
    add("gutz72-fp32-608", "honeycomb", 6, 6, "fp32", 608, 8.0)
    # the same model in the split-precision mode, half the chains, shorter projection
    add("gutz72-bf16x3-304", "honeycomb", 6, 6, "bf16x3", 304, 4.0)
    # the same model in FP64: production where single precision is not trusted
    add("gutz72-fp64-304", "honeycomb", 6, 6, "fp64", 304, 4.0)
    # the variational (g, M_N) scan, 242 chains of 72 / 162 / 288 sites in one launch
    add("scan-fp32-242", "scan", 12, 12, "fp32", 242, 2.0)
    # sign study of the doped square lattice, 256 chains
    add("doped64-fp32-256", "square", 8, 8, "fp32", 256, 12.0, g=0.3, M_N=0.0)
    # spinless t-V chains: bond fields, one species
    add("tv72-fp32-304", "tv", 6, 6, "fp32", 304, 4.0, U=1.6, g=0.3, M_N=0.24)
    # chains too large for an SM's shared memory, one per SM, split-precision products
    add("large162-bf16x3-152", "honeycomb", 9, 9, "bf16x3", 152, 4.0)
    # one large chain swept by the whole GPU
    add("spread648-fp32-1", "honeycomb", 18, 18, "fp32", 1, 2.0, spread=True)
    add("spread288-fp64-1", "honeycomb", 12, 12, "fp64", 1, 4.0, spread=True)
    # G of given fields in FP64 (post-processing of stored configurations)
    add("green72-fp64", "honeycomb", 6, 6, "fp64", 1, 8.0, use="green")
    return out


def _sites(case):
    return case["Lx"] * case["Ly"] * (1 if case["model"] == "square" else 2)


def _slices(case):
    return int(round(case["two_theta"] / 0.1))


def estimate(case):
    """Seconds of one pass, roughly (measured rates of a chain per slice, and waves of chains over 152 SMs)."""
    N, rows = _sites(case), _slices(case) + 2
    if case["spread"]:
        return case["chains"] * rows * ((N / 648) ** 1.5 * 3.3e-3 if case["prec"] != "fp64" else (N / 288) ** 2 * 1.8e-3)
    if case["prec"] == "fp64":
        per, at_once = 1.4e-4 + 2.1e-3 * (N / 72) ** 3, 608
    else:
        per, at_once = 3e-4 * (N / 72) ** 2.5, 304 if N < 128 else 152
    return per * rows * math.ceil(case["chains"] / at_once)


def draw(rng):
    """One more use of the same ranges: lattices of 8 to 648 sites (Lx and Ly apart, odd ones too), one to 608 chains, every precision."""
    while True:
        kind = rng.choice(["honeycomb", "honeycomb", "honeycomb", "square", "tv", "spread", "green"])
        prec = rng.choice(["fp64", "fp32", "fp32", "bf16x3"])
        use = "green" if kind == "green" else "sweep"
        sites = math.exp(rng.uniform(math.log(8), math.log(648 if kind == "spread" else 288)))
        if kind == "spread":
            sites = max(sites, 64)
        if kind == "square":
            Lx = Ly = 8
        else:
            Lx = max(2, int(round(math.sqrt(sites / 2) * rng.uniform(0.7, 1.4))))
            Ly = max(2, int(round(sites / 2 / Lx)))
        model = kind if kind in ("square", "tv") else "honeycomb"
        chains = 1 if use == "green" else int(round(math.exp(rng.uniform(0, math.log(3 if kind == "spread" else 608)))))
        n_stab = rng.choice([5, 5 if kind == "spread" else 10]) if prec == "fp64" else rng.choice([1, 2, 2])
        two_theta = 0.1 * 2 * n_stab * int(round(math.exp(rng.uniform(math.log(2), math.log(120))) / (2 * n_stab)))
        if kind == "tv":
            par = {"U": round(rng.uniform(1.2, 1.8), 3), "g": round(rng.uniform(0, 0.4), 3), "M_N": round(rng.uniform(0.1, 0.3), 3)}
        else:
            par = {"U": round(rng.uniform(3.5, 4.0), 3), "g": round(rng.uniform(0, 0.8), 3),
                   "M_N": 0.0 if kind == "square" else round(rng.uniform(0.05, 0.3), 3)}
        c = _case(model, Lx, Ly, prec, chains, round(two_theta, 6), use=use, n_stab=n_stab, spread=kind == "spread", **par)
        if two_theta > 0 and _sites(c) <= 648 and estimate(c) <= MAX_SECONDS:
            return c


def _specs(case):
    n = case["chains"]
    if case["model"] == "scan":
        return workloads.variational_grid(case["two_theta"])[:n]
    kw = dict(U=case["U"], dtau=0.1, two_theta=case["two_theta"], g=case["g"], M_N=case["M_N"])
    if case["model"] == "square":
        kw.update(kind=workloads.SQUARE, tp=-0.2, n_up=28, n_dn=28)
    elif case["model"] == "tv":
        kw.update(kind=workloads.HONEYCOMB_TV, n_up=-1, n_dn=0)
    else:
        kw.update(kind=workloads.HONEYCOMB)
    return [workloads.ChainSpec(Lx=case["Lx"], Ly=case["Ly"], **kw)] * n


class _State:
    def __init__(self, case, ctx, fields, species):
        self.case, self.ctx, self.fields, self.species = case, ctx, fields, species
        self.kind = np.float64 if case["prec"] == "fp64" else np.float32

    def __del__(self):
        self.ctx.close()


def prepare(case, seed):
    specs = _specs(case)
    ctx = pqmc.Context(specs, prec=PRECISION[case["prec"]], seed=seed, n_stab=case["n_stab"], spread=1 if case["spread"] else 0)
    fields = workloads.random_fields(specs[0], seed) if case["use"] == "green" else None
    return _State(case, ctx, fields, 1 if case["model"] == "tv" else 2)


def run(state):
    ctx, kind = state.ctx, state.kind
    if state.case["use"] == "green":
        ctx.set_fields(state.fields)
        return {"G": [ctx.green(0, s).astype(kind) for s in range(state.species)], "weight": ctx.weight().astype(kind)}
    ctx.sweep(1, measure=True)
    out = {"records": ctx.last_records().astype(kind)}
    if state.case["chains"] <= FEW:
        out["G"] = [ctx.green(c, s).astype(kind) for c in range(state.case["chains"]) for s in range(state.species)]
        out["fields"] = [ctx.fields(c) for c in range(state.case["chains"])]
    return out


def work(case):
    """Per chain and sweep: the fields, G and the stack blocks of each species in and out once; the wrap (two products per slice), the
    delayed updates at an acceptance of one half, the stack products, and per stabilisation the QR, the overlap, its inverse and G."""
    ts = 8 if case["prec"] == "fp64" else 4
    total_b = total_f = 0.0
    for s in _specs(case):
        N, Lt = s.n_sites, s.n_slices
        n = s.n_up if s.n_up >= 0 else N // 2
        sp = 1 if case["model"] == "tv" else 2
        nb = Lt // case["n_stab"] + 1
        stab = 2 * n * n * (N - n / 3) + 2 * n * n * N + 2 * n ** 3 + 2 * n * n * N + 2 * N * N * n
        if case["use"] == "green":
            total_b += (Lt + 2) * s.n_fields + sp * N * N * 8 + 2 * N * N * ts + sp * N * n * 8
            total_f += sp * (Lt * 2 * N * N * n + nb * 2 * n * n * (N - n / 3) + stab)
        else:
            total_b += 2 * (Lt + 2) * s.n_fields + 2 * sp * N * N * ts + 2 * sp * nb * N * n * 8
            total_f += sp * (Lt * 4 * N ** 3 + (Lt + 2) * N ** 3 + Lt * 2 * N * N * n + nb * stab)
    return {"bytes": total_b, "flops": total_f}


# ---------------------------------------------------------------------------
# The same results in plain NumPy, FP64: whole sweeps of one FP64 chain, and G of given fields.


def _philox(c0, c1, c2, c3, seed):
    """Philox4x32-10 over arrays of 32-bit counter words (Salmon et al., SC'11)."""
    m = np.uint64(0xFFFFFFFF)
    c = [np.asarray(x, np.uint64) * np.ones_like(np.asarray(c0, np.uint64)) for x in (c0, c1, c2, c3)]
    k0, k1 = seed & 0xFFFFFFFF, seed >> 32
    for _ in range(10):
        p, q = np.uint64(0xD2511F53) * c[0], np.uint64(0xCD9E8D57) * c[2]
        c = [(q >> np.uint64(32)) ^ c[1] ^ np.uint64(k0), q & m, (p >> np.uint64(32)) ^ c[3] ^ np.uint64(k1), p & m]
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return c


class _Plain:
    """One honeycomb Hubbard chain: slices 0 and Lt + 1 carry the Gutzwiller fields, 1 .. Lt the interaction's."""

    def __init__(self, case):
        Lx, Ly = case["Lx"], case["Ly"]
        self.N, self.Lt, self.U = 2 * Lx * Ly, _slices(case), case["U"]
        N = self.N
        K = np.zeros((N, N))
        for y in range(Ly):
            for x in range(Lx):
                a = 2 * (x + Lx * y)
                for b in (a + 1, 2 * ((x - 1) % Lx + Lx * y) + 1, 2 * (x + Lx * ((y - 1) % Ly)) + 1):
                    K[a, b] -= 1.0
                    K[b, a] -= 1.0
        self.K, self.eps = K, np.where(np.arange(N) % 2 == 0, 1.0, -1.0)
        w, v = np.linalg.eigh(K)
        self.Em, self.Ep = (v * np.exp(-0.1 * w)) @ v.T, (v * np.exp(0.1 * w)) @ v.T
        m = max(case["M_N"], 1e-4)
        self.P = [np.linalg.eigh(K + sg * m * np.diag(self.eps))[1][:, : N // 2] for sg in (1, -1)]
        self.kappa = [float(np.arccosh(np.exp(x / 2))) for x in (0.1 * self.U, case["g"])]

    def edge(self, tau):
        return tau in (0, self.Lt + 1)

    def diag(self, f, tau, sp):
        return np.exp((1 - 2 * sp) * self.kappa[1 if self.edge(tau) else 0] * f[tau])

    def green(self, f, tau):
        """G at tau (-1: before slice 0) of both spins, and (log |det|, sign) of each spin's weight."""
        G, weight = [], []
        for sp in (0, 1):
            R, log, sign = self.P[sp], 0.0, 1.0
            L = self.P[sp]

            def factor(M):
                q, r = np.linalg.qr(M)
                d = np.diag(r)
                return q, float(np.log(np.abs(d)).sum()), float(np.prod(np.sign(d)))

            for t in range(0, tau + 1):
                M = self.diag(f, t, sp)[:, None] * R
                R, a, b = factor(M if self.edge(t) else self.Em @ M)
                log, sign = log + a, sign * b
            for t in range(self.Lt + 1, tau, -1):
                M = L if self.edge(t) else self.Em @ L
                L, a, b = factor(self.diag(f, t, sp)[:, None] * M)
                log, sign = log + a, sign * b
            O = L.T @ R
            s, a = np.linalg.slogdet(O)
            G.append(np.eye(self.N) - R @ np.linalg.solve(O, L.T))
            weight += [log + a, sign * s]
        return G, weight

    def sweep_up(self, seed):
        """The first sweep of chain 0 from its own initial fields: the record, G and the fields after it."""
        N, Lt = self.N, self.Lt
        tau, site = np.divmod(np.arange((Lt + 2) * N), N)
        f = np.where(_philox(site, tau, 0xFFFFFFFF, 0, seed)[2] & np.uint64(1), 1, -1).astype(np.int8).reshape(Lt + 2, N)
        x = _philox(site, tau, 0, 0, seed)
        u = (((x[0] << np.uint64(21)) | (x[1] >> np.uint64(11))).astype(np.float64) * 2.0 ** -53).reshape(Lt + 2, N)
        G, weight = self.green(f, -1)
        running, record = weight[1] * weight[3], None
        for t in range(Lt + 2):
            for i in range(N):
                d = [math.exp(-2 * (1 - 2 * sp) * self.kappa[1 if self.edge(t) else 0] * f[t, i]) - 1 for sp in (0, 1)]
                r = [1 + d[sp] * (1 - G[sp][i, i]) for sp in (0, 1)]
                if u[t, i] < abs(r[0] * r[1]):
                    for sp in (0, 1):
                        col = -G[sp][:, i]
                        col[i] += 1.0
                        G[sp] -= np.outer(col * (d[sp] / r[sp]), G[sp][i].copy())
                    f[t, i] = -f[t, i]
                    running *= math.copysign(1.0, r[0] * r[1])
            if t % 5 == 0 and t <= Lt:
                G, weight = self.green(f, t)
            else:
                for sp in (0, 1):
                    v = self.diag(f, t, sp)
                    A = v[:, None] * G[sp] / v[None, :]
                    G[sp] = A if self.edge(t) else self.Em @ A @ self.Ep
            if t == Lt // 2:
                record = self.record(*self.green(f, t), running)
        return record, G, f

    def record(self, G, weight, running):
        N, dens = self.N, [1 - np.diag(g) for g in G]
        c = [np.eye(N) - g.T for g in G]
        kin = sum(float((self.K * x).sum()) for x in c) / N
        docc = float((dens[0] * dens[1]).sum()) / N
        ee = np.outer(self.eps, self.eps)
        s = (float((self.eps * (dens[0] - dens[1])).sum()) ** 2 + sum(float((ee * c[k] * G[k]).sum()) for k in (0, 1))) / (4.0 * N * N)
        return [weight[1] * weight[3], kin + self.U * docc, docc, kin, running, s]


def exact(case, seed):
    """Honeycomb Hubbard chains only.  Sweeps: one FP64 chain (in FP32 a proposal whose ratio lies next to its uniform may go the other
    way than in 64 bits, and the trajectories part), up to what NumPy does in a few seconds."""
    if case["model"] != "honeycomb" or _sites(case) > 162:
        return None
    plain = _Plain(case)
    if case["use"] == "green":
        G, weight = plain.green(_given_fields(case, seed), -1)
        return {"G": G, "weight": np.array(weight)}
    if case["prec"] != "fp64" or case["chains"] > 1 or (plain.Lt + 2) * plain.N > 12000:
        return None
    record, G, fields = plain.sweep_up(seed)
    return {"records": np.array([record]), "G": G, "fields": [fields]}


def _given_fields(case, seed):
    """The fields that prepare() hands over: uniform +-1, from the seed."""
    shape = (_slices(case) + 2, _sites(case))
    return np.random.default_rng(seed).choice(np.array([-1, 1], dtype=np.int8), size=shape)
