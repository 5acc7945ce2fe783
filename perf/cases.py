"""Performance cases of the library: the work a user's program has it do, through its public entry points.

A case is a dict of plain values:

    kind     "steps"    flbm_step(n) on one lattice (a run between two looks at it)
             "sampled"  a measuring loop: flbm_sample and n steps, repeated, then flbm_fetch_samples
             "stats"    flbm_stats of the state in hand
             "batch"    an ensemble: n steps of every lattice, then one sample of each, fetched
    lattice  "d2q9", "d3q27", "d3q27_iso", "d3q19"; nx, ny, nz the periodic box
    storage  "fp32", "bf16", "fp16" deviations
    rates    "paper" (the shear modes at `omega`, every other mode at 1), "uniform" (every
             non-conserved mode at `omega`), "modes" (a rate of its own for every mode)
    raw      the raw-moment collision (fluctuating BGK when the rates are uniform)
    tuned    the program calls autotune once it has its lattice, as long runs do

The state a lattice starts from is a thermal one: the equilibrium at density 1 and a uniform drift,
plus the equilibrium fluctuations of every population (variance 3 kBT w_i), drawn from the seed.
Populations are returned as the caller's own device buffer (stored deviations f_i - w_i). Statistics
are means of single-precision quantities, so they are handed on in that type.
"""
import math

import numpy as np
import torch

import paper_2602_16486_gb300 as fl

LATTICES = {"d2q9": fl.FLBM_D2Q9, "d3q27": fl.FLBM_D3Q27, "d3q27_iso": fl.FLBM_D3Q27_ISO, "d3q19": fl.FLBM_D3Q19}
STORAGES = {"fp32": (fl.FLBM_FP32, torch.float32), "bf16": (fl.FLBM_BF16, torch.bfloat16),
            "fp16": (fl.FLBM_FP16, torch.float16)}


def _case(name, kind, lattice, dims, storage="fp32", rates="paper", omega=1.6, kbt=1e-4, steps=1, samples=0,
          drift=0.0, raw=False, tuned=False):
    c = dict(name=name, kind=kind, lattice=lattice, nx=dims[0], ny=dims[1], nz=dims[2], storage=storage, rates=rates,
             omega=omega, kbt=kbt, steps=steps, samples=samples, drift=drift, raw=raw, tuned=tuned)
    if name is None:
        del c["name"]
    return c


def _batch(name, lattices, mix, steps):
    c = dict(name=name, kind="batch", lattices=lattices, mix=mix, steps=steps)
    if name is None:
        del c["name"]
    return c


def listed():
    third = 1.0 / 3000.0
    return [
        # A small 2-D box with one rate for every mode, stepped from a driver program: launches count.
        _case("d2q9_64_uniform", "steps", "d2q9", (64, 64, 1), rates="uniform", omega=1.25, steps=100),
        # The 2-D equipartition run of the paper: a sample every 20 steps, gathered in blocks.
        _case("d2q9_200_sampled", "sampled", "d2q9", (200, 200, 1), omega=1.25, kbt=third, steps=20, samples=10),
        # The statistics ensemble's 2-D member near the over-relaxation limit.
        _case("d2q9_512", "steps", "d2q9", (512, 512, 1), omega=1.9, steps=50),
        # A large 2-D box in 16-bit storage, tuned.
        _case("d2q9_4096_bf16", "steps", "d2q9", (4096, 4096, 1), storage="bf16", omega=1.5, steps=4, tuned=True),
        # The comparison scheme, fluctuating BGK, on a 3-D box.
        _case("d3q27_96_bgk", "steps", "d3q27", (96, 96, 96), rates="uniform", omega=1.25, steps=10, raw=True),
        # The paper's second anisotropic box (odd rows) with its sampling interval.
        _case("d3q27_25x50x100_sampled", "sampled", "d3q27", (25, 50, 100), omega=1.25, kbt=third, steps=20, samples=5),
        # The statistics ensemble's 3-D member.
        _case("d3q27_64", "steps", "d3q27", (64, 64, 64), omega=1.98, steps=50),
        # The headline run: drift, FP32, statistics every 10 steps.
        _case("d3q27_256_headline", "sampled", "d3q27", (256, 256, 256), steps=10, samples=1, drift=0.05, tuned=True),
        # The same box with 16-bit deviations (the precision sweep).
        _case("d3q27_256_fp16", "steps", "d3q27", (256, 256, 256), storage="fp16", steps=10, tuned=True),
        # The reduced velocity set at full size.
        _case("d3q19_256", "steps", "d3q19", (256, 256, 256), steps=10, tuned=True),
        # The ensemble of 256 mixed lattices: 100 steps, then one sample of every member.
        _batch("batch_256_mixed", 256, 0, 100),
        # Watching a run: the statistics of a large state on their own.
        _case("stats_d3q27_256", "stats", "d3q27", (256, 256, 256), drift=0.05),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges."""
    kind = rng.choice(("steps", "steps", "steps", "sampled", "stats", "batch"))
    if kind == "batch":
        return _batch(None, _log(rng, 16, 256), rng.randrange(1, 10 ** 6), _log(rng, 5, 60))
    lattice = rng.choice(("d2q9", "d3q27", "d3q27", "d3q27_iso", "d3q19"))
    if lattice == "d2q9":
        dims = (_log(rng, 32, 4096), _log(rng, 32, 4096), 1)
    else:
        dims = (_log(rng, 12, 256), _log(rng, 12, 256), _log(rng, 12, 256))
    raw = lattice in ("d2q9", "d3q27") and rng.random() < 0.15
    rates = rng.choice(("paper", "paper", "uniform", "modes"))
    sites = dims[0] * dims[1] * dims[2]
    steps = max(1, min(_log(rng, 1, 100), 6 * 10 ** 7 // sites))
    samples = rng.randint(1, 8) if kind == "sampled" else 0
    if samples:
        steps = max(1, min(steps, 6 * 10 ** 7 // (sites * samples)))
    if kind == "stats":
        steps = 1
    # The comparison scheme breaks down towards rate 2 and at high temperature: it is used below.
    omega, kbt = rng.uniform(0.6, 1.4 if raw else 1.98), rng.choice((0.0, 1e-5, 1e-4, 1.0 / 3000.0, 1e-3))
    return _case(None, kind, lattice, dims, storage=rng.choice(("fp32", "fp32", "bf16", "fp16")), rates=rates,
                 omega=round(omega, 3), kbt=min(kbt, 1e-4) if raw else kbt,
                 steps=steps, samples=samples, drift=rng.choice((0.0, 0.05)), raw=raw, tuned=rng.random() < 0.5)


# ---- the lattices' tables and a thermal state ------------------------------------------------
D2Q9 = [(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)]
D3Q27 = ([(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1)]
         + [(x, y, 0) for y in (1, -1) for x in (1, -1)] + [(x, 0, z) for z in (1, -1) for x in (1, -1)]
         + [(0, y, z) for z in (1, -1) for y in (1, -1)]
         + [(x, y, z) for z in (1, -1) for y in (1, -1) for x in (1, -1)])


def _velocities(lattice):
    if lattice == "d2q9":
        return [(x, y, 0) for x, y in D2Q9]
    return D3Q27[:19] if lattice == "d3q19" else D3Q27


def _weights(lattice):
    n = [sum(abs(a) for a in c) for c in _velocities(lattice)]
    table = {"d2q9": (4 / 9, 1 / 9, 1 / 36), "d3q19": (1 / 3, 1 / 18, 1 / 36)}.get(lattice, (8 / 27, 2 / 27, 1 / 54, 1 / 216))
    return [table[k] for k in n]


def _lam(case):
    q = len(_velocities(case["lattice"]))
    d = 2 if q == 9 else 3
    if case["rates"] == "modes":
        lam = 1.0 + 0.6 * np.sin(1.0 + 1.7 * np.arange(q)) * (case["omega"] - 1.0)
    elif case["rates"] == "uniform":
        lam = np.full(q, case["omega"])
    else:
        lam = np.ones(q)
        lam[[4, 5] if d == 2 else [7, 8, 9]] = case["omega"]
        if case["lattice"] == "d3q27_iso":
            lam[[5, 6]] = case["omega"]
    lam[:d + 1] = 1.0
    return lam


def _thermal_state(case, seed, device):
    """Stored deviations of a thermal state, [q][z][y][x], in the storage type."""
    vel, w = _velocities(case["lattice"]), _weights(case["lattice"])
    shape = (case["nz"], case["ny"], case["nx"])
    gen = torch.Generator(device=device)
    gen.manual_seed(int(seed))
    u = (case["drift"], 0.4 * case["drift"], 0.0)
    out = torch.empty((len(vel),) + shape, dtype=STORAGES[case["storage"]][1], device=device)
    for i, c in enumerate(vel):
        cu = sum(a * b for a, b in zip(c, u))
        eq = w[i] * (3.0 * cu + 4.5 * cu * cu - 1.5 * sum(a * a for a in u))
        noise = torch.randn(shape, generator=gen, device=device, dtype=torch.float32)
        out[i] = eq + math.sqrt(3.0 * max(case["kbt"], 1e-6) * w[i]) * noise
    return out


def _ensemble(case, seed):
    """The members of a batch: geometry from the case, physics and noise seeds from the seed."""
    rng, phys = np.random.default_rng(case["mix"]), np.random.default_rng(seed)
    specs = []
    for j in range(case["lattices"]):
        d3 = rng.random() < 0.5
        lo, hi = (16, 64) if d3 else (32, 256)
        side = int(round(np.exp(rng.uniform(np.log(lo), np.log(hi)))))
        lam = np.ones(27 if d3 else 9)
        lam[[7, 8, 9] if d3 else [4, 5]] = 1.0 / phys.uniform(0.51, 2.0)
        specs.append(dict(lattice=fl.FLBM_D3Q27 if d3 else fl.FLBM_D2Q9, dims=(side, side, side if d3 else 1), lam=lam,
                          kBT=float(np.exp(phys.uniform(np.log(1e-5), np.log(1e-3)))), rho0=1.0,
                          seed=int(phys.integers(1 << 40))))
    return specs


_stream = None


def prepare(case, seed):
    global _stream
    if _stream is None:
        _stream = torch.cuda.Stream()
    if case["kind"] == "batch":
        specs = _ensemble(case, seed)
        batch = fl.Batch(specs, cuda_stream=_stream.cuda_stream)
        for i in range(len(specs)):
            batch.lattice(i).init_uniform((0.02, 0.01, 0.0), 1e-2, seed)
        batch.autotune(4)
        batch.sync()
        return dict(case=case, batch=batch)
    code, dims = LATTICES[case["lattice"]], (case["nx"], case["ny"], case["nz"])
    storage, dtype = STORAGES[case["storage"]]
    buf = torch.empty((len(_velocities(case["lattice"])),) + dims[::-1], dtype=dtype, device="cuda")
    torch.cuda.synchronize()
    lat = fl.Lattice(code, dims, _lam(case), case["kbt"], 1.0, seed, storage, cuda_stream=_stream.cuda_stream,
                     dev_buf=buf.data_ptr(), dev_buf_bytes=buf.numel() * buf.element_size())
    if case["raw"]:
        lat.collision = fl.FLBM_COLLISION_RAW
    lat.sync()
    buf.copy_(_thermal_state(case, seed, "cuda"))
    torch.cuda.synchronize()
    if case["tuned"]:
        lat.autotune(10)
    return dict(case=case, lattice=lat, f=buf)


def _records(samples):
    """Samples as arrays: [mass, momentum], [<u>, <uu>], <k>, <k k^T>."""
    return dict(conserved=np.array([np.append(s["mass"], s["mom"]) for s in samples], dtype=np.float32),
                velocity=np.array([np.append(s["u_mean"], s["uu"]) for s in samples], dtype=np.float32),
                modes=np.array([s["k_mean"] for s in samples], dtype=np.float32),
                covariance=np.array([s["k_cov"] for s in samples], dtype=np.float32))


def run(state):
    case = state["case"]
    if case["kind"] == "batch":
        batch = state["batch"]
        batch.step(case["steps"])
        members = [batch.lattice(i) for i in range(len(batch))]
        for lat in members:
            lat.sample()
        got = [lat.fetch_samples(1)[0] for lat in members]
        return {d: _records([s for s in got if s["q"] == q]) for d, q in (("d2q9", 9), ("d3q27", 27))
                if any(s["q"] == q for s in got)}
    lat = state["lattice"]
    if case["kind"] == "steps":
        lat.step(case["steps"])
        return dict(f=state["f"])
    if case["kind"] == "stats":
        return _records([lat.stats()])
    for _ in range(case["samples"]):
        lat.sample()
        lat.step(case["steps"])
    return dict(f=state["f"], **_records(lat.fetch_samples()))


def _site_bytes(case):
    """(bytes of one site's populations, floating-point operations of one site's update)."""
    q = len(_velocities(case["lattice"]))
    normals = (q - (3 if q == 9 else 4)) if case["kbt"] > 0 else 0
    return q * (4 if case["storage"] == "fp32" else 2), 14 * q + 40 * normals


def work(case):
    """Every step reads and writes each population once; a sample reads each once."""
    if case["kind"] == "batch":
        nbytes = flops = 0
        for s in _ensemble(case, 0):
            d3 = s["lattice"] == fl.FLBM_D3Q27
            sites, q = s["dims"][0] ** (3 if d3 else 2), 27 if d3 else 9
            nbytes += sites * q * 4 * (2 * case["steps"] + 1)
            flops += sites * case["steps"] * (14 * q + 40 * (23 if d3 else 6))
        return dict(bytes=nbytes, flops=flops)
    sites = case["nx"] * case["ny"] * case["nz"]
    b, f = _site_bytes(case)
    gram = 2 * (16 if case["lattice"] == "d2q9" else 32) ** 2
    if case["kind"] == "stats":
        return dict(bytes=sites * b, flops=sites * gram)
    reps = max(1, case["samples"])
    return dict(bytes=sites * b * (2 * case["steps"] * reps + case["samples"]),
                flops=sites * (f * case["steps"] * reps + gram * case["samples"]))


# ---- the same in 64 bits, in plain torch ------------------------------------------------------
# Tensor orders (x, y, z) of the D3Q27 modes: M_v is the product of 1, c and c^2 - 1/3 along the axes.
D3Q27_MODES = [(0, 0, 0), (1, 0, 0), (0, 1, 0), (0, 0, 1), (2, 0, 0), (0, 2, 0), (0, 0, 2), (1, 1, 0), (1, 0, 1),
               (0, 1, 1), (2, 1, 0), (2, 0, 1), (1, 2, 0), (1, 0, 2), (0, 1, 2), (0, 2, 1), (1, 1, 1), (2, 2, 0),
               (2, 0, 2), (0, 2, 2), (1, 1, 2), (1, 2, 1), (2, 1, 1), (2, 1, 2), (2, 2, 1), (1, 2, 2), (2, 2, 2)]
NORM1 = (1.0, 1.0 / 3.0, 2.0 / 9.0)


def _d3q19_basis(x, y, z):
    r = x * x + y * y + z * z
    one = torch.ones_like(x)
    return [one, x, y, z, r - 1, 3 * x * x - r, y * y - z * z, x * y, y * z, x * z, x * (3 * r - 5), y * (3 * r - 5),
            z * (3 * r - 5), x * (y * y - z * z), y * (z * z - x * x), z * (x * x - y * y), 3 * r * r - 6 * r + 1,
            (2 * r - 3) * (3 * x * x - r), (2 * r - 3) * (y * y - z * z)]


D3Q19_NORMS = [1, 1 / 3, 1 / 3, 1 / 3, 2 / 3, 4 / 3, 4 / 9, 1 / 9, 1 / 9, 1 / 9, 2 / 3, 2 / 3, 2 / 3, 2 / 9, 2 / 9, 2 / 9,
               2, 4 / 3, 4 / 9]


def _norms(lattice):
    if lattice == "d2q9":
        return [1, 1 / 3, 1 / 3, 4 / 9, 4 / 9, 1 / 9, 2 / 27, 2 / 27, 4 / 81]
    if lattice == "d3q19":
        return D3Q19_NORMS
    b = [NORM1[i] * NORM1[j] * NORM1[k] for i, j, k in D3Q27_MODES]
    if lattice == "d3q27_iso":
        b[4:7] = [2 / 3, 4 / 9, 4 / 3]
    return b


def _normals(site, step, seed, count):
    """`count` standard normals of every site: Philox4x32-10 keyed on (seed; site, step, block), Box-Muller."""
    mask, out = 0xFFFFFFFF, []

    def mul(a, m):  # high and low words of a 32 x 32 bit product, in signed 64-bit arithmetic
        lo, hi = a * (m & 0xFFFF), a * (m >> 16)
        s = (lo >> 16) + hi
        return s >> 16, ((s & 0xFFFF) << 16) | (lo & 0xFFFF)

    for block in range((count + 3) // 4):
        x, y = site.clone(), torch.full_like(site, step & mask)
        z, w = torch.full_like(site, (step >> 32) & mask), torch.full_like(site, block)
        k0, k1 = seed & mask, (seed >> 32) & mask
        for _ in range(10):
            h0, l0 = mul(x, 0xD2511F53)
            h1, l1 = mul(z, 0xCD9E8D57)
            x, y, z, w = h1 ^ y ^ k0, l1, h0 ^ w ^ k1, l0
            k0, k1 = (k0 + 0x9E3779B9) & mask, (k1 + 0xBB67AE85) & mask
        u = [((v >> 9).double() + 0.5) * 2.0 ** -23 for v in (x, y, z, w)]
        for a, b in ((u[0], u[1]), (u[2], u[3])):
            r, t = torch.sqrt(-2.0 * torch.log(a)), 2.0 * math.pi * b
            out += [r * torch.cos(t), r * torch.sin(t)]
    return out[:count]


class _Exact:
    """One lattice in 64 bits: populations f[q] over the flattened sites."""

    def __init__(self, case, seed):
        self.case, self.seed, self.lam = case, int(seed), _lam(case)
        self.lat, self.vel, self.w = case["lattice"], _velocities(case["lattice"]), _weights(case["lattice"])
        self.shape = (case["nz"], case["ny"], case["nx"])
        self.device = "cuda" if torch.cuda.is_available() else "cpu"
        self.d = 2 if self.lat == "d2q9" else 3
        self.f = [x.double() + w for x, w in zip(_thermal_state(case, seed, self.device), self.w)]
        self.t = 0

    def macros(self):
        rho = sum(self.f)
        j = [sum(c[a] * f for c, f in zip(self.vel, self.f)) for a in range(3)]
        j = [x if torch.is_tensor(x) else torch.zeros_like(rho) for x in j]
        return rho, j, [x / rho for x in j]

    def forward(self, u):
        """Moments in the paper's order about the velocity u (u = 0: raw moments)."""
        if self.lat == "d3q19":
            k = [torch.zeros_like(self.f[0]) for _ in range(19)]
            for c, f in zip(self.vel, self.f):
                for v, m in enumerate(_d3q19_basis(c[0] - u[0], c[1] - u[1], c[2] - u[2])):
                    k[v] = k[v] + m * f
            return k
        t = dict(zip(self.vel, self.f))
        for axis in range(self.d):
            new = {}
            for c in t:
                if c[axis] != 0:
                    continue
                m, o, p = (t[c[:axis] + (s,) + c[axis + 1:]] for s in (-1, 0, 1))
                s0, s1, s2 = m + o + p, p - m, p + m
                ua = u[axis]
                got = (s0, s1 - ua * s0, s2 - 2 * ua * s1 + ua * ua * s0 - s0 / 3)
                for order in range(3):
                    new[c[:axis] + (order,) + c[axis + 1:]] = got[order]
            t = new
        if self.d == 2:
            a, b = t[2, 0, 0], t[0, 2, 0]
            return [t[0, 0, 0], t[1, 0, 0], t[0, 1, 0], a + b, a - b, t[1, 1, 0], t[2, 1, 0], t[1, 2, 0], t[2, 2, 0]]
        k = [t[m] for m in D3Q27_MODES]
        if self.lat == "d3q27_iso":
            a, b, c = k[4:7]
            k[4:7] = [a + b + c, a - b, a + b - 2 * c]
        return k

    def inverse(self, k, u):
        if self.lat == "d3q19":
            rows = []
            for c in self.vel:
                rows.append(torch.stack([m.reshape(-1) for m in _d3q19_basis(c[0] - u[0], c[1] - u[1], c[2] - u[2])], -1))
            mat = torch.stack(rows, -1)  # [site, mode, velocity]
            sol = torch.linalg.solve(mat, torch.stack([x.reshape(-1) for x in k], -1))
            return [sol[:, i].reshape(self.shape) for i in range(19)]
        if self.d == 2:
            a, b = (k[3] + k[4]) / 2, (k[3] - k[4]) / 2
            t = {(0, 0, 0): k[0], (1, 0, 0): k[1], (0, 1, 0): k[2], (2, 0, 0): a, (0, 2, 0): b, (1, 1, 0): k[5],
                 (2, 1, 0): k[6], (1, 2, 0): k[7], (2, 2, 0): k[8]}
        else:
            k = list(k)
            if self.lat == "d3q27_iso":
                tr, p, q = k[4:7]
                s = (2 * tr + q) / 3
                k[4:7] = [(s + p) / 2, (s - p) / 2, (tr - q) / 3]
            t = dict(zip(D3Q27_MODES, k))
        for axis in range(self.d):
            new = {}
            for o in t:
                if o[axis] != 0:
                    continue
                k0, k1, k2 = (t[o[:axis] + (s,) + o[axis + 1:]] for s in range(3))
                ua = u[axis]
                s1 = k1 + ua * k0
                s2 = k2 + k0 / 3 + 2 * ua * s1 - ua * ua * k0
                for c, v in ((-1, (s2 - s1) / 2), (0, k0 - s2), (1, (s2 + s1) / 2)):
                    new[o[:axis] + (c,) + o[axis + 1:]] = v
            t = new
        return [t[c] for c in self.vel]

    def step(self):
        rho, _, u = self.macros()
        zero = [torch.zeros_like(rho)] * 3
        raw = self.case["raw"]
        k = self.forward(zero if raw else u)
        if raw:  # the raw moments of the product equilibrium
            m = [(1.0, x, x * x) for x in u]
            t = {(a, b, c): rho * m[0][a] * m[1][b] * m[2][c] for a in range(3) for b in range(3)
                 for c in (range(3) if self.d == 3 else range(1))}
            if self.d == 2:
                a, b = t[2, 0, 0], t[0, 2, 0]
                keq = [rho, None, None, a + b, a - b, t[1, 1, 0], t[2, 1, 0], t[1, 2, 0], t[2, 2, 0]]
            else:
                keq = [t[o] for o in D3Q27_MODES]
        first, q = self.d + 1, len(self.vel)
        kbt, lam, norm = self.case["kbt"], self.lam, _norms(self.lat)
        if kbt > 0:
            site = torch.arange(rho.numel(), device=self.device).reshape(self.shape)
            eta = _normals(site, self.t, self.seed, q - first)
        post = list(k)
        post[0] = rho
        if not raw:
            post[1:first] = [torch.zeros_like(rho)] * self.d
        for v in range(first, q):
            x = (1.0 - lam[v]) * k[v]
            if raw:
                x = x + lam[v] * keq[v]
            if kbt > 0:
                x = x + torch.sqrt(rho * (kbt * lam[v] * (2.0 - lam[v]) * norm[v] * 3.0)) * eta[v - first]
            post[v] = x
        f = self.inverse(post, zero if raw else u)
        self.f = [torch.roll(x, (c[2], c[1], c[0]), (0, 1, 2)) for c, x in zip(self.vel, f)]
        self.t += 1

    def stored(self):
        """Deviations as the in-place streaming keeps them: after an odd number of steps slot i of
        site y holds the opposite population of site y - c_i."""
        out = []
        for i, c in enumerate(self.vel):
            if self.t % 2 == 0:
                out.append(self.f[i] - self.w[i])
            else:
                opp = self.vel.index(tuple(-a for a in c))
                out.append(torch.roll(self.f[opp], (c[2], c[1], c[0]), (0, 1, 2)) - self.w[i])
        return torch.stack(out)

    def record(self):
        rho, j, u = self.macros()
        k, n = self.forward(u), rho.numel()
        for v in range(1, self.d + 1):
            k[v] = torch.zeros_like(rho)
        k = torch.stack([x.reshape(-1) for x in k])
        pairs = ((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2))
        return dict(mass=rho.sum().item(), mom=np.array([x.sum().item() for x in j]),
                    u_mean=np.array([x.mean().item() for x in u]),
                    uu=np.array([(u[a] * u[b]).mean().item() for a, b in pairs]),
                    k_mean=k.mean(1).cpu().numpy(), k_cov=(k @ k.T / n).cpu().numpy())


def exact(case, seed):
    if case["kind"] == "batch":
        return None  # hundreds of lattices: minutes in plain torch
    sites = case["nx"] * case["ny"] * case["nz"]
    updates = sites * (1 if case["kind"] == "stats" else case["steps"] * max(1, case["samples"]))
    gpu = torch.cuda.is_available()
    most = 4e6 if case["lattice"] == "d3q19" and case["kind"] != "stats" else 1e9
    if updates > (most if gpu else most / 200) or (case["lattice"] == "d3q19" and sites > 5e5 and case["kind"] != "stats"):
        return None
    with torch.no_grad():
        e = _Exact(case, seed)
        if case["kind"] == "stats":
            return _double([e.record()])
        got = []
        for _ in range(max(1, case["samples"])):
            if case["samples"]:
                got.append(e.record())
            for _ in range(case["steps"]):
                e.step()
        out = dict(f=e.stored())
        return dict(out, **_double(got)) if got else out


def _double(samples):
    return dict(conserved=np.array([np.append(s["mass"], s["mom"]) for s in samples]),
                velocity=np.array([np.append(s["u_mean"], s["uu"]) for s in samples]),
                modes=np.array([s["k_mean"] for s in samples]), covariance=np.array([s["k_cov"] for s in samples]))
