"""The work that is timed: what a program that uses this library has it do.

A case names one job and its sizes. prepare() makes what such a program holds
before the job (a lattice, a batch or a server, with page-locked host arrays
for the states it reads back), run() is the job: steps through the public
entry points, then the state and the correlations the program is after, and
exact() is the same job in 64-bit torch, written from the paper's equations
without the package's code.

Populations come back as flb_get_populations returns them. Correlation sums of
FP32 and FP16-store lattices are formed from FP32 products and partials, and
structure factors of FP32 lattices from FP32 transforms, so those are returned
as float32 arrays, which hold all their digits; FP64 lattices return float64.
"""
import math

import numpy as np
import torch

from paper_1204_6734_gb300 import flb, inputs

SHEAR_BULK_GHOST = (1.0, 0.8, 1.0)


# ---------------------------------------------------------------------------
# Cases
# ---------------------------------------------------------------------------

def lattice_case(name, Lx, Ly, basis, steps, every=1, precision="fp32", ux0=0.1, spectrum=0):
    """One lattice: `steps` steps, the correlations sampled every `every` steps
    (0: not at all, a thermalisation), the structure factors every `spectrum`."""
    c = {"kind": "lattice", "Lx": Lx, "Ly": Ly, "basis": basis, "precision": precision, "ux0": ux0,
         "steps": steps, "every": every, "spectrum": spectrum}
    return {"name": name, **c} if name else c


def copies_case(name, side, n, basis, steps):
    """n copies of a small side x side lattice, a third of them at each of three
    u_x0, in one batch, and the pooled correlations of each u_x0."""
    c = {"kind": "copies", "side": side, "n": n, "basis": basis, "steps": steps}
    return {"name": name, **c} if name else c


def ensemble_case(name, n, lo, hi, basis, steps, tile="mixed", sizes=3):
    """n uneven replicas with sides in [lo, hi] (their `sizes`-th set), in one batch."""
    c = {"kind": "ensemble", "n": n, "lo": lo, "hi": hi, "basis": basis, "steps": steps, "tile": tile, "sizes": sizes}
    return {"name": name, **c} if name else c


def serving_case(name, n, lo, hi, shortest, longest, chunk=16, sizes=5):
    """n requests (the `sizes`-th trace) submitted to a running server, and all their results."""
    c = {"kind": "serving", "n": n, "lo": lo, "hi": hi, "shortest": shortest, "longest": longest, "chunk": chunk,
         "sizes": sizes}
    return {"name": name, **c} if name else c


def listed():
    return [
        # the paper's own lattice: a run's block of steps between two looks at its state
        lattice_case("paper_21", 21, 21, "local", 500),
        # the spectra of Figs. 19 to 24: correlations every step, structure factors every 5
        lattice_case("spectrum_64", 64, 64, "local", 500, ux0=0.2, spectrum=5),
        # an uneven lattice of ordinary size in the table f-norm
        lattice_case("table_300x130", 300, 130, "lut", 500, ux0=0.2),
        # a larger one before its sampling starts
        lattice_case("thermal_1000x750", 1000, 750, "local", 500, every=0),
        # the Hermite norm, the form that existing codes use, sampled as it runs
        lattice_case("hermite_2048", 2048, 2048, "standard", 300),
        # the lattice the library is measured on
        lattice_case("fnorm_4096", 4096, 4096, "local", 200),
        # the paper's 21 x 21 statistics: pooled copies at several velocities
        copies_case("copies_21", 21, 384, "local", 2000),
        # a parameter study: uneven replicas in the tiling that the tuner picks for them
        ensemble_case("ensemble_48", 48, 64, 1024, "local", 150),
        # requests to a server, each a lattice of its own size and length
        serving_case("serving_24", 24, 32, 512, 100, 800),
        # the 64-bit reference runs: the small one that results are checked on, and an uneven larger one
        lattice_case("fp64_32", 32, 32, "local", 300, precision="fp64"),
        lattice_case("fp64_400x300", 400, 300, "local", 100, precision="fp64", ux0=0.2),
        # the precision study's half-width store
        lattice_case("fp16_2000x1500", 2000, 1500, "local", 200, precision="fp16dev", ux0=0.2),
    ]


def log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["lattice", "lattice", "lattice", "spectrum", "copies", "ensemble", "serving", "fp64", "fp16"])
    basis = rng.choice(["local", "local", "standard", "lut"])
    ux0 = rng.choice([0.0, 0.05, 0.1, 0.2, 0.3])
    if kind == "copies":
        side = log_int(rng, 9, 64)
        n = 3 * log_int(rng, 8, 160)
        return copies_case(None, side, n, basis, max(100, min(2000, int(4e8 / (n * side * side)))))
    if kind == "ensemble":
        lo = log_int(rng, 16, 128)
        return ensemble_case(None, log_int(rng, 4, 64), lo, log_int(rng, 2 * lo, 1024), basis, rng.randint(40, 150),
                             rng.choice(["mixed", "64x12", "128x4"]), sizes=rng.randint(10, 10 ** 6))
    if kind == "serving":
        return serving_case(None, log_int(rng, 4, 32), 32, log_int(rng, 64, 512), 50, log_int(rng, 100, 800),
                            rng.choice([8, 16, 32]), sizes=rng.randint(10, 10 ** 6))
    if kind == "fp64":
        Lx, Ly = log_int(rng, 16, 512), log_int(rng, 16, 512)
        return lattice_case(None, Lx, Ly, basis, max(10, min(500, int(1.5e7 / (Lx * Ly)))), precision="fp64", ux0=ux0,
                            every=rng.choice([1, 1, 10, 0]))
    if kind == "spectrum":
        if rng.random() < 0.6:
            Lx, Ly = 2 ** rng.randint(4, 11), 2 ** rng.randint(4, 11)
        else:
            Lx, Ly = log_int(rng, 16, 300), log_int(rng, 16, 300)
        return lattice_case(None, Lx, Ly, basis, max(20, min(500, int(5e8 / (Lx * Ly)))), ux0=ux0,
                            spectrum=rng.choice([2, 5, 10]))
    top = 4096 if kind == "lattice" else 2500
    Lx, Ly = log_int(rng, 16, top), log_int(rng, 16, top)
    steps = max(20, min(500, int((3e9 if kind == "lattice" else 1e9) / (Lx * Ly))))
    return lattice_case(None, Lx, Ly, basis, steps, ux0=ux0, every=rng.choice([1, 1, 1, 10, 0]),
                        precision="fp32" if kind == "lattice" else "fp16dev")


# ---------------------------------------------------------------------------
# What a case consists of
# ---------------------------------------------------------------------------

def lattices(c, seed):
    """The parameters of every lattice of a case."""
    if c["kind"] == "lattice":
        return [inputs.LatticeParams(c["Lx"], c["Ly"], 1.0, c["ux0"], 0.0, 1e-4, inputs.omega_groups(*SHEAR_BULK_GHOST),
                                     c["basis"], c["precision"], seed=seed)]
    if c["kind"] == "copies":
        return [inputs.LatticeParams(c["side"], c["side"], 1.0, (0.05, 0.1, 0.2)[3 * r // c["n"]], 0.0, 1e-4,
                                     inputs.omega_groups(*SHEAR_BULK_GHOST), c["basis"], "fp32",
                                     seed=(seed << 16) + r, replica=r) for r in range(c["n"])]
    if c["kind"] == "ensemble":
        ps = inputs.replica_ensemble(c["n"], c["sizes"], c["lo"], c["hi"], c["basis"])
        for r, p in enumerate(ps):
            p.seed = (seed << 16) + r
        return ps
    return [q.params for q in requests(c, seed)]


def requests(c, seed):
    g = np.random.Generator(np.random.PCG64(c["sizes"]))
    rs = inputs.serving_requests(c["n"], seed=c["sizes"], lo=c["lo"], hi=c["hi"])
    for q in rs:   # shorter runs than the trace's, so that a job is a fraction of a second
        q.steps = int(g.integers(c["shortest"], c["longest"] + 1))
        q.warmup = q.steps // 10
        q.params.seed = (seed << 16) + q.rid
    return rs


def pinned(shape):
    return torch.empty(shape, dtype=torch.float64, pin_memory=True).numpy()


def prepare(case, seed):
    c = dict(case)
    ps = lattices(c, seed)
    s = {"case": c, "ps": ps}
    if c["kind"] == "lattice":
        lat = flb.Lattice(ps[0])
        lat.set_sampling(0, c["every"])
        if c["spectrum"]:
            lat.set_structure_sampling(0, c["spectrum"])
        s["lattice"], s["f"] = lat, pinned((9, c["Ly"], c["Lx"]))
    elif c["kind"] == "serving":
        s["requests"] = requests(c, seed)
        pool = sum(flb.flb_batch_replica_bytes(p) for p in ps)
        s["server"] = flb.Server("local", pool_bytes=pool, max_slots=c["n"], chunk_steps=c["chunk"])
    else:
        b = flb.Batch(ps, tile=c.get("tile"))
        b.set_sampling(0, 1)
        s["batch"] = b
        ends = 9 * np.cumsum([p.nodes for p in ps])   # the replicas' states one after the other
        s["f"] = pinned((int(ends[-1]),))
        s["views"] = [v.reshape(9, p.Ly, p.Lx) for v, p in zip(np.split(s["f"], ends[:-1]), ps)]
    return s


def single(a):
    return np.asarray(a, dtype=np.float32)


def run(state):
    c, ps = state["case"], state["ps"]
    if c["kind"] == "lattice":
        lat, keep = state["lattice"], np.asarray if c["precision"] == "fp64" else single
        lat.step(c["steps"])
        out = {"f": flb.flb_get_populations(lat.h, c["Lx"], c["Ly"], state["f"])}
        if c["every"]:
            Cff, CMM, mean, n = lat.correlations("standard" if c["basis"] == "standard" else "local")
            out.update(Cff=keep(Cff), CMM=keep(CMM), mean=keep(mean), samples=n)
        if c["spectrum"]:
            S_rho, S_jx, R, n = lat.structure_factors()
            out.update(S_rho=keep(S_rho), S_jx=keep(S_jx), R=R if c["precision"] == "fp64" else R.astype(np.complex64),
                       spectra=n)
        return out
    if c["kind"] == "serving":
        s = state["server"]
        first = [s.submit(q.params, q.steps, q.warmup, q.every) for q in state["requests"]][0]
        done = sorted(s.drain(), key=lambda r: r["id"])
        return {"id": np.array([r["id"] - first for r in done]), "status": np.array([r["status"] for r in done]),
                "samples": np.array([r["n_samples"] for r in done]),
                "S1": single([r["S1"] for r in done]), "S2": single([r["S2"] for r in done])}
    b = state["batch"]
    b.step(c["steps"])
    if c["kind"] == "copies":
        basis = "standard" if c["basis"] == "standard" else "local"
        k = c["n"] // 3
        got = [b.correlations(list(range(j * k, (j + 1) * k)), basis) for j in range(3)]
        out = {"Cff": single([g[0] for g in got]), "CMM": single([g[1] for g in got]),
               "mean": single([g[2] for g in got]), "samples": np.array([g[3] for g in got])}
    else:
        sums = [b.raw_sums(r) for r in range(c["n"])]
        out = {"S1": single([g[0] for g in sums]), "S2": single([g[1] for g in sums]),
               "samples": np.array([g[2] for g in sums])}
    for r, p in enumerate(ps):
        flb.flb_batch_get_populations(b.h, r, p.Lx, p.Ly, state["views"][r])
    out["f"] = state["f"]
    return out


def work(case):
    """Bytes: the populations read and written once in each step, in the store's
    width, and the state given back as doubles; operations of a step as the
    paper's equations take them (basis, moments, relaxation, noise)."""
    c = case
    if c["kind"] == "serving":
        node_steps = sum(q.params.nodes * q.steps for q in requests(c, 1))
        return {"bytes": 72.0 * node_steps, "flops": 800.0 * node_steps}
    nodes = sum(p.nodes for p in lattices(c, 1))
    width = {"fp64": 8, "fp32": 4, "fp16dev": 2}[c.get("precision", "fp32")]
    ops = 300.0 if c["basis"] == "standard" else 800.0
    return {"bytes": 18.0 * width * nodes * c["steps"] + 72.0 * nodes, "flops": ops * nodes * c["steps"]}


# ---------------------------------------------------------------------------
# The same jobs in 64 bits
# ---------------------------------------------------------------------------

VX = (0, 1, 0, -1, 0, 1, -1, -1, 1)
VY = (0, 0, 1, 0, -1, 1, 1, -1, -1)
WEIGHTS = (4 / 9,) + (1 / 9,) * 4 + (1 / 36,) * 4


def hermite_rows():
    """The nine rows of the Hermite moments (rho, j_x, j_y, Pi_xx-yy, Pi_xy,
    Pi_xx+yy, q_x, q_y, epsilon), orthonormal under the weights w_i: Gram-Schmidt
    of the monomials 1, v_x, v_y, v_x^2 - v_y^2, v_x v_y, v_x^2 + v_y^2,
    v_x v^2, v_y v^2, v^4 under the weights, with the paper's signs."""
    vx, vy, w = np.array(VX, float), np.array(VY, float), np.array(WEIGHTS)
    v2 = vx * vx + vy * vy
    rows = []
    for m in (np.ones(9), vx, vy, vx * vx - vy * vy, vx * vy, v2, vx * v2, vy * v2, v2 * v2):
        for r in rows:
            m = m - (m * r * w).sum() * r
        rows.append(m / math.sqrt((m * m * w).sum()))
    return np.array(rows)


def equilibrium(ux, uy):
    """f_i^0(1, u), stacked over i."""
    out = []
    for i in range(9):
        uv = VX[i] * ux + VY[i] * uy
        out.append(WEIGHTS[i] * (1 + 3 * uv + 4.5 * uv * uv - 1.5 * (ux * ux + uy * uy)))
    return torch.stack(out)


def philox_normals(node, step, replica, key_lo, key_hi):
    """Six standard normals of each node: Philox4x32-10 of (node, step, replica,
    0), six 21-bit fields of its 128 bits, three Box-Muller pairs."""
    low = 0xFFFFFFFF
    c = [node, torch.full_like(node, step), replica, torch.zeros_like(node)]
    k0, k1 = key_lo, key_hi
    for _ in range(10):
        p0, p1 = c[0] * 0xD2511F53, c[2] * 0xCD9E8D57   # modulo 2^64
        c = [((p1 >> 32) & low) ^ c[1] ^ k0, p1 & low, ((p0 >> 32) & low) ^ c[3] ^ k1, p0 & low]
        k0, k1 = (k0 + 0x9E3779B9) & low, (k1 + 0xBB67AE85) & low
    m21 = (1 << 21) - 1
    a, b = c[0] | (c[1] << 32), c[2] | (c[3] << 32)   # two 64-bit halves
    k = [a & m21, (a >> 21) & m21, (a >> 42) & m21, ((a >> 63) & 1) | ((b & ((1 << 20) - 1)) << 1),
         (b >> 20) & m21, (b >> 41) & m21]
    n = []
    for p in range(3):
        r = torch.sqrt(-2 * torch.log((k[2 * p] + 1).double() * 2.0 ** -21))
        t = 2 * math.pi * (k[2 * p + 1].double() * 2.0 ** -21)
        n += [r * torch.cos(t), r * torch.sin(t)]
    return torch.stack(n)


def solve_collision(P, W, Y, D_of):
    """P^T L^-T D with L the Cholesky factor of P diag(W) P^T (the f-norm basis is
    L^-1 P), D = D_of(L^-1 Y)."""
    N = W.shape[1]
    pairs = torch.stack([P[a] * P[b] for a in range(9) for b in range(9)])
    L = (pairs @ W).reshape(9, 9, N)
    for j in range(9):
        if j:
            L[j:, j] -= (L[j:, :j] * L[j, :j]).sum(1)
        L[j, j] = torch.sqrt(L[j, j])
        L[j + 1:, j] /= L[j, j].clone()
    y = Y.clone()
    for j in range(9):
        if j:
            y[j] -= (L[j, :j] * y[:j]).sum(0)
        y[j] /= L[j, j]
    z = D_of(y)
    for j in range(8, -1, -1):
        if j < 8:
            z[j] -= (L[j + 1:, j] * z[j + 1:]).sum(0)
        z[j] /= L[j, j]
    return P.T @ z


class Plain:
    """Lattices of one basis stepped together in 64 bits, their nodes in one row."""

    def __init__(self, ps):
        self.dev = dev = "cuda" if torch.cuda.is_available() else "cpu"
        self.ps, self.basis = ps, ps[0].basis
        f64 = {"dtype": torch.float64, "device": dev}
        self.P = torch.tensor(hermite_rows(), **f64)
        sizes = [p.nodes for p in ps]
        self.at = np.concatenate([[0], np.cumsum(sizes)])
        rep = torch.repeat_interleave(torch.arange(len(ps), device=dev), torch.tensor(sizes, device=dev))
        self.rep = rep

        def of(values, **kw):
            return torch.tensor(values, device=dev, **kw)[rep]
        self.node = torch.arange(int(self.at[-1]), device=dev) - of(self.at[:-1].tolist())
        Lx, Ly = of([p.Lx for p in ps]), of([p.Ly for p in ps])
        x, y = self.node % Lx, self.node // Lx
        base = self.node.new_tensor(self.at[:-1])[rep]
        self.pull = [base + (x - VX[i]) % Lx + ((y - VY[i]) % Ly) * Lx for i in range(9)]
        self.key = (of([p.seed & 0xFFFFFFFF for p in ps]), of([p.seed >> 32 for p in ps]), of([p.replica for p in ps]))
        om = torch.tensor([list(p.omega[3:]) for p in ps], **f64).T[:, rep]
        kT = of([p.kT for p in ps], dtype=torch.float64)
        self.om, self.amp = om, torch.sqrt(kT * om * (2 - om))
        self.c = torch.stack([equilibrium(torch.tensor(p.ux0, **f64), torch.tensor(p.uy0, **f64)) * p.rho0
                              for p in ps]).T[:, rep].contiguous()
        self.f = self.c.clone()   # pre-collision state f_i(x, t)
        self.w = torch.tensor(WEIGHTS, **f64)
        self.t = 0
        self.vx, self.vy = torch.tensor(VX, **f64), torch.tensor(VY, **f64)

    def step(self):
        g, P = self.f, self.P
        rho = g.sum(0)
        ux, uy = (self.vx @ g) / rho, (self.vy @ g) / rho
        Y = P @ (g - rho * equilibrium(ux, uy))
        xi = torch.sqrt(rho) * self.amp * philox_normals(self.node, self.t, self.key[2], self.key[0], self.key[1])

        def increments(y):
            z = torch.zeros_like(y)
            z[3:] = xi - self.om * y[3:]
            return z
        if self.basis == "standard":
            f = g + self.w[:, None] * (P.T @ increments(Y))
        else:
            if self.basis == "lut":   # the basis at the nearest velocity of the 51 x 51 table
                ux, uy = (torch.floor(50 * u + 25.5) / 50 - 0.5 for u in (ux, uy))
            W = equilibrium(ux, uy)
            f = g + W * solve_collision(P, W, Y, increments)
        self.f = torch.stack([f[i][self.pull[i]] for i in range(9)])
        self.t += 1

    def sums(self, r):
        d = (self.f - self.c)[:, self.at[r]:self.at[r + 1]]
        return d.sum(1), d @ d.T

    def state(self, r):
        return self.f[:, self.at[r]:self.at[r + 1]].reshape(9, self.ps[r].Ly, self.ps[r].Lx).cpu()


def measured(S1, S2, n, p, basis):
    """<df df>, <dM dM> in the Hermite rows or the f-norm at u0, and the mean deviation."""
    mean = S1 / n
    C = S2 / n - np.outer(mean, mean)
    B = hermite_rows()
    if basis != "standard":
        W = equilibrium(torch.tensor(p.ux0, dtype=torch.float64), torch.tensor(p.uy0, dtype=torch.float64)).numpy()
        B = np.linalg.solve(np.linalg.cholesky((B * W) @ B.T), B)
    return C, B @ C @ B.T, mean


def exact(case, seed):
    c = case
    ps = lattices(c, seed)
    if c["kind"] == "serving":
        rs = requests(c, seed)
        last, rates = max(q.steps for q in rs), [(q.warmup, q.steps, q.every) for q in rs]
    else:
        every = 1 if c["kind"] != "lattice" else c["every"]
        last, rates = c["steps"], [(0, c["steps"], every)] * len(ps)
    if last * (3e-3 + 3e-9 * sum(p.nodes for p in ps)) > 20:   # seconds, about
        return None
    m = Plain(ps)
    K = len(ps)
    S1 = torch.zeros(K, 9, dtype=torch.float64, device=m.dev)
    S2 = torch.zeros(K, 81, dtype=torch.float64, device=m.dev)
    spectra = {}
    ij = [(i, j) for i in range(9) for j in range(9)]
    due = [torch.zeros(K, dtype=torch.float64) for _ in range(last)]
    for r, (warm, stop, every) in enumerate(rates):
        if every:
            for t in range(warm, stop, every):
                due[t][r] = 1.0
    for t in range(last):
        take = due[t].to(m.dev)
        if K == 1:
            if take.item():
                a, b = m.sums(0)
                S1[0] += a
                S2[0] += b.reshape(81)
        elif take.any():
            d = m.f - m.c
            S1 += take[:, None] * torch.zeros(K, 9, dtype=d.dtype, device=m.dev).index_add_(0, m.rep, d.T.contiguous())
            for k, (i, j) in enumerate(ij):
                if i <= j:
                    v = take * torch.zeros(K, dtype=d.dtype, device=m.dev).index_add_(0, m.rep, d[i] * d[j])
                    S2[:, 9 * i + j] += v
                    if i != j:
                        S2[:, 9 * j + i] += v
        if c.get("spectrum") and t % c["spectrum"] == 0:
            d = (m.f - m.c).reshape(9, c["Ly"], c["Lx"])
            r = torch.fft.fft2(d.sum(0))
            a = torch.fft.fft2(torch.einsum("i,ixy->xy", m.vx, d))
            b = torch.fft.fft2(torch.einsum("i,ixy->xy", m.vy, d))
            for key, v in (("S_rho", (r * r.conj()).real), ("S_jx", (a * a.conj()).real), ("R", a * b.conj())):
                spectra[key] = spectra.get(key, 0) + v
        m.step()
    S1, S2 = S1.cpu().numpy(), S2.cpu().numpy().reshape(K, 9, 9)
    nodes = np.array([p.nodes for p in ps])
    n = nodes * np.array([int(sum(due[t][r] for t in range(last))) for r in range(K)])
    if c["kind"] == "serving":
        return {"id": None, "status": None, "samples": n, "S1": S1, "S2": S2}
    if c["kind"] == "lattice":
        out = {"f": m.state(0)}
        if c["every"]:
            C, M, mean = measured(S1[0], S2[0], n[0], ps[0], c["basis"])
            if c["precision"] == "fp16dev":   # the store's rounding of the conserved sums is all of it
                mean = None
            out.update(Cff=C, CMM=M, mean=mean, samples=int(n[0]))
        if c["spectrum"]:
            k = (c["steps"] + c["spectrum"] - 1) // c["spectrum"]
            out.update({key: (v / (k * ps[0].rho0)).cpu().numpy() for key, v in spectra.items()}, spectra=k)
        return out
    f = np.concatenate([m.state(r).numpy().reshape(-1) for r in range(K)])
    if c["kind"] == "copies":
        k = K // 3
        got = [measured(S1[j * k:(j + 1) * k].sum(0), S2[j * k:(j + 1) * k].sum(0), n[j * k:(j + 1) * k].sum(), ps[j * k],
                        c["basis"]) for j in range(3)]
        return {"Cff": np.stack([g[0] for g in got]), "CMM": np.stack([g[1] for g in got]),
                "mean": np.stack([g[2] for g in got]), "samples": np.array([n[j * k:(j + 1) * k].sum() for j in range(3)]),
                "f": f}
    return {"S1": S1, "S2": S2, "samples": n, "f": f}
