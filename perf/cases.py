"""Performance cases: the calls that a user of the package makes, over the sizes
that they are made at.

listed() gives the named cases, draw() more of the same ranges; prepare() makes
what a program holds before the call, run() is one pass through the public entry
points and work() the bytes and operations the call cannot do without.  exact()
restates the computation in 64-bit torch without the package: FFT moving average
for the fields, and for the solves the same Picard iteration with direct
(block-tridiagonal) linear solves in place of multigrid.
"""
import functools
import math

import numpy as np
import torch

import paper_1903_08741_gb300 as R

MAP_ALPHAS = [0.2 * k for k in range(1, 21)]
MAP_NS = [1.1 + 0.1 * k for k in range(10)] + [2.2 + 0.2 * k for k in range(10)]
PICARD_PER_STEP, CYCLES_PER_PICARD = 25, 5          # typical, for work() only


def listed():
    return [
        # the fields of the 32^2 x 64 plain Monte Carlo run: the smallest draw, bound by launches
        {"name": "fields_32_s64", "kind": "fields", "nx": 32, "nz": 32, "samples": 64, "nu": 0.0},
        # the fields of the 128^2 batch, an eighth of the 4096 samples
        {"name": "fields_128_s512", "kind": "fields", "nx": 128, "nz": 128, "samples": 512, "nu": 0.0},
        # five van Genuchten soil fields (Matern Phi_1) as the fine / coarse couples of an MLMC level
        {"name": "soil_pair_64_s512", "kind": "soil_pair", "nx": 64, "nz": 64, "samples": 512, "nu": 1.0},
        # the whole 32^2 x 64, 10-step plain Monte Carlo run: fewer samples than SMs
        {"name": "mc_32_s64_fp64", "kind": "solve", "nx": 32, "nz": 32, "samples": 64, "steps": 10, "dt": 0.01,
         "mixed": False, "scale": 1.0, "host": False},
        # the 128^2 batch (2 of its 20 steps, two full waves of samples), FP64: the headline throughput
        {"name": "mc_128_s608_fp64", "kind": "solve", "nx": 128, "nz": 128, "samples": 608, "steps": 2, "dt": 0.005,
         "mixed": False, "scale": 1.0, "host": False},
        # the same batch with FP32 V-cycles inside FP64 defect correction
        {"name": "mc_128_s608_mixed", "kind": "solve", "nx": 128, "nz": 128, "samples": 608, "steps": 2, "dt": 0.005,
         "mixed": True, "scale": 1.0, "host": False},
        # the (alpha, n) cost map: infiltration, van Genuchten-Mualem, W(2,2), 32^2, thousands of tiny solves
        {"name": "vg_map_32_s4096", "kind": "vg", "nx": 32, "nz": 32, "samples": 4096, "steps": 6, "dt": 1.0 / 64,
         "mixed": False, "thetas": False},
        # one sample alone, at the 64^2 MLMC level's nonlinearity: what trying out one soil costs, latency only
        {"name": "one_64_fp64", "kind": "solve", "nx": 64, "nz": 64, "samples": 1, "steps": 10, "dt": 0.01,
         "mixed": False, "scale": 0.6, "host": False},
        # the finest MLMC level's few samples (256^2, dt = 0.1 / 80), mixed precision
        {"name": "finest_256_s24_mixed", "kind": "solve", "nx": 256, "nz": 256, "samples": 24, "steps": 2,
         "dt": 0.1 / 80, "mixed": True, "scale": 1.0, "host": False},
        # a grid that is no power of two (coarsest 6 x 5), fields and results in host memory, continuation 0.8
        {"name": "ragged_96x80_host", "kind": "solve", "nx": 96, "nz": 80, "samples": 200, "steps": 2, "dt": 0.01,
         "mixed": False, "scale": 0.8, "host": True},
        # forward and backward of the differentiable QoI (32 KL coefficients)
        {"name": "adjoint_64_s48", "kind": "adjoint", "nx": 64, "nz": 64, "samples": 48, "steps": 6, "dt": 0.005,
         "modes": 32, "mixed": False, "ckpt": 3},
        # a whole three-level MLMC estimate with parametric continuation
        {"name": "mlmc_16_32_64", "kind": "mlmc", "n0": 16, "levels": 3, "samples": 2048, "ratio": 4, "steps": 5,
         "coupling": 2, "mixed": False},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _side(rng, lo, hi):
    """A side k 2^m, k = 4 ... 7."""
    while True:
        n = rng.choice([4, 5, 6, 7]) << rng.randint(0, 6)
        if lo <= n <= hi:
            return n


def _coarsens(nx, nz):
    while nx % 2 == 0 and nz % 2 == 0 and nx * nz > 4:
        nx, nz = nx // 2, nz // 2
    return nx * nz <= 64


def draw(rng):
    kind = rng.choice(["fields", "fields", "soil_pair", "solve", "solve", "solve", "solve", "vg", "adjoint", "mlmc"])
    if kind in ("fields", "soil_pair"):
        nx, nz = (1 << rng.randint(4, 8) for _ in range(2))
        if max(nx, nz) > 4 * min(nx, nz):
            nx = nz
        most = min(8192, (512 * 128 * 128 if kind == "fields" else 512 * 64 * 64) // (nx * nz))
        return {"kind": kind, "nx": nx, "nz": nz, "samples": _log_int(rng, 1, max(1, most)),
                "nu": rng.choice([0.0, 1.0, 0.5])}
    if kind == "mlmc":
        return {"kind": kind, "n0": rng.choice([8, 16]), "levels": rng.choice([2, 3]),
                "samples": _log_int(rng, 200, 2000), "ratio": 4, "steps": rng.randint(2, 5),
                "coupling": rng.choice([0, 1, 2]), "mixed": rng.random() < 0.5}
    while True:
        nx, nz = _side(rng, 8, 256), _side(rng, 8, 256)
        if rng.random() < 0.5:
            nx = nz
        if max(nx, nz) <= 4 * min(nx, nz) and _coarsens(nx, nz):
            break
    # cell-steps of a pass on one SM, at most those of the largest listed batch
    steps = rng.randint(1, 10)
    cap = {"solve": 90000, "vg": 60000, "adjoint": 12000}[kind]
    while nx * nz * steps > cap and steps > 1:
        steps -= 1
    if nx * nz * steps > cap:
        nx = nz = 32
    most = max(1, int(200 * cap / (nx * nz * steps)))
    case = {"kind": kind, "nx": nx, "nz": nz, "samples": _log_int(rng, 1, min(most, 8192)), "steps": steps,
            "mixed": rng.random() < 0.4}
    if kind == "solve":
        case.update(dt=rng.choice([0.01, 0.005, 0.1 / 80]), scale=rng.choice([0.4, 0.8, 1.0]),
                    host=rng.random() < 0.2)
    elif kind == "vg":
        case.update(dt=1.0 / 64, thetas=rng.random() < 0.5)
    else:
        case.update(dt=0.005, modes=rng.choice([8, 32, 64]), ckpt=rng.randint(1, 10))
    return case


# ---------------------------------------------------------------- inputs
def _gaussian_pairs(count, nz, nx, gen, corr=0.3):
    """Two independent Gaussian fields [count, nz, nx] of exponential covariance
    (circulant embedding on twice the grid, spacing 1/nz)."""
    h = 1.0 / nz
    a = torch.arange(2 * nx, device="cuda", dtype=torch.float64)
    b = torch.arange(2 * nz, device="cuda", dtype=torch.float64)
    a, b = torch.minimum(a, 2 * nx - a) * h, torch.minimum(b, 2 * nz - b) * h
    lam = torch.fft.fft2(torch.exp(-torch.sqrt(a[None, :] ** 2 + b[:, None] ** 2) / corr)).real.clamp_min(0.0)
    out = []
    for k in range(0, count, 128):
        m = min(128, count - k)
        y = torch.randn((2, m, 2 * nz, 2 * nx), device="cuda", dtype=torch.float64, generator=gen)
        z = torch.fft.ifft2(torch.sqrt(lam) * torch.fft.fft2(torch.complex(y[0], y[1])))[:, :nz, :nx]
        out.append((z.real.contiguous(), z.imag.contiguous()))
    return torch.cat([o[0] for o in out]), torch.cat([o[1] for o in out])


def _phi(g):
    return 0.5 * torch.erfc(-g / math.sqrt(2.0))


def _kl_basis(nz, nx, modes):
    """The leading modes of the separable exponential covariance on the grid's
    cells (corr. length 0.2), sqrt(eigenvalue) folded in."""
    def line(n, h):
        x = torch.arange(n, dtype=torch.float64) * h
        w, v = torch.linalg.eigh(torch.exp(-(x[:, None] - x[None, :]).abs() / 0.2))
        w, v = w.flip(0).clamp_min(0.0), v.flip(1)
        v = v * torch.sign(v[v.abs().argmax(0), torch.arange(n)])
        return w, v
    wx, vx = line(nx, 1.0 / nz)
    wz, vz = line(nz, 1.0 / nz)
    pairs = torch.argsort((wz[:, None] * wx[None, :]).reshape(-1), descending=True, stable=True)[:modes]
    J, I = pairs // nx, pairs % nx
    B = torch.sqrt(wz[J] * wx[I])[:, None, None] * vz.T[J][:, :, None] * vx.T[I][:, None, :]
    return B.contiguous().cuda()


_kl_basis = functools.lru_cache(maxsize=8)(_kl_basis)


def _inputs(c, seed):
    """The arrays of a solve: a dict of [S, nz, nx] float64 CUDA tensors."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    S, nz, nx = c["samples"], c["nz"], c["nx"]
    lk, g = _gaussian_pairs(S, nz, nx, gen)
    if c["kind"] == "solve":
        return {"lnKs": lk, "alpha": 0.5 + 1.5 * _phi(g)}
    if c["kind"] == "adjoint":
        xi = torch.randn((S, c["modes"]), device="cuda", dtype=torch.float64, generator=gen)
        return {"xi": xi, "alpha": 0.5 + 1.5 * _phi(g), "basis": _kl_basis(nz, nx, c["modes"])}
    # cost map: one (alpha, n) pair per sample, walked through the table from a random start
    k = torch.arange(S) + int(torch.randint(0, 400, (1,), device="cuda", generator=gen))
    pa = torch.tensor(MAP_ALPHAS, dtype=torch.float64)[(k * 7) % 20].cuda()
    pn = torch.tensor(MAP_NS, dtype=torch.float64)[(k * 3 + k // 20) % len(MAP_NS)].cuda()
    d = {"lnKs": lk + math.log(0.2), "alpha": pa[:, None, None].expand(S, nz, nx).contiguous(),
         "n": pn[:, None, None].expand(S, nz, nx).contiguous()}
    if c["thetas"]:
        u, v = _gaussian_pairs(S, nz, nx, gen)
        d["theta_s"], d["theta_r"] = 0.45 + 0.1 * _phi(u), 0.045 + 0.01 * _phi(v)
    return d


def _model(c, seed):
    if c["nu"] == 1.0:
        return R.FieldModel.phi1(seed=seed)
    if c["nu"] == 0.5:
        return R.FieldModel.phi2(seed=seed)
    return R.FieldModel(seed=seed)


def _problem(c):
    prec = R.MIXED if c["mixed"] else R.FP64
    if c["kind"] == "vg":
        return R.Problem.infiltration(nx=c["nx"], nz=c["nz"], nsteps=c["steps"], dt=c["dt"], precision=prec)
    return R.Problem(nx=c["nx"], nz=c["nz"], nsteps=c["steps"], dt=c["dt"], precision=prec)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "fields":
        return {"case": case, "model": _model(case, seed)}
    if kind == "soil_pair":
        return {"case": case, "model": R.soil_field_model(3.0, _model(case, seed)), "soil": R.SoilModel()}
    if kind == "mlmc":
        n = [max(2, case["samples"] // case["ratio"] ** l) for l in range(case["levels"])]
        return {"case": case, "cfg": R.MlmcConfig(
            nsamples=tuple(n), n0=case["n0"], steps0=case["steps"], coupling=case["coupling"],
            problem=R.Problem(precision=R.MIXED if case["mixed"] else R.FP64), model=R.FieldModel(seed=seed))}
    state = {"case": case, "problem": _problem(case), **_inputs(case, seed)}
    if case.get("host"):
        state["lnKs"], state["alpha"] = state["lnKs"].cpu().numpy(), state["alpha"].cpu().numpy()
    if kind == "adjoint":
        state["xi"].requires_grad_(True)
        state["ones"] = torch.ones(case["samples"], dtype=torch.float64, device="cuda")
    return state


def run(state):
    c = state["case"]
    kind = c["kind"]
    if kind == "fields":
        return R.sample_fields(c["nx"], c["nz"], c["samples"], state["model"])
    if kind == "soil_pair":
        return R.sample_soil_pair(c["nx"], c["nz"], c["samples"], state["model"], state["soil"])
    if kind == "mlmc":
        r = R.mlmc_estimate(state["cfg"])
        return {k: np.asarray(r[k]) for k in ("estimate", "mean", "var", "mean_f", "var_f", "mean_c", "var_c", "n",
                                              "failed")}
    if kind == "adjoint":
        qoi = R.RichardsQoI.apply(state["xi"], state["alpha"], state["basis"], state["problem"], 1.0, c["ckpt"])
        return qoi, torch.autograd.grad(qoi, state["xi"], state["ones"])[0]
    if kind == "vg":
        qoi, p, status, _, _ = R.solve_soil(state["problem"], state["lnKs"], state["alpha"], state["n"],
                                            state.get("theta_s"), state.get("theta_r"), want_p=True)
    elif c["host"]:
        qoi, p, status, _, _ = R.solve_batch_host(state["problem"], state["lnKs"], state["alpha"], c["scale"],
                                                  want_p=True)
        p[np.isnan(qoi)] = np.nan                       # a failed sample has no head, as it has no QoI
        return qoi, p, status
    else:
        qoi, p, status, _, _ = R.solve_batch(state["problem"], state["lnKs"], state["alpha"], c["scale"],
                                             want_p=True)
    return qoi, p.masked_fill_(torch.isnan(qoi)[:, None, None], math.nan), status


def work(case):
    kind = case["kind"]
    if kind == "mlmc":
        cells = sum((case["samples"] / case["ratio"] ** l) * (case["n0"] << l) ** 2 * 1.25 for l in
                    range(case["levels"]))
        csteps = sum((case["samples"] / case["ratio"] ** l) * (case["n0"] << l) ** 2 * (case["steps"] << l) * 1.125
                     for l in range(case["levels"]))
        io = 8.0 * 9 * case["levels"]
    else:
        cells = case["nx"] * case["nz"] * case["samples"]
        csteps = cells * case.get("steps", 0)
        arrays = {"fields": 2, "soil_pair": 6.25, "solve": 3, "vg": 4 + 2 * case.get("thetas", False),
                  "adjoint": 1}[kind]
        io = 8.0 * arrays * cells
    # FFT moving average on the doubled torus (two real fields in one complex transform)
    packs = {"fields": 1.0, "soil_pair": 3.75, "mlmc": 1.25}.get(kind, 0.0)
    side = case.get("nx", 64) * case.get("nz", 64) * 4.0
    flops = packs * 4 * cells * (10.0 * math.log2(side) + 60.0)
    # a V-cycle is about 55 and a Picard iteration about 51 operations a cell; the adjoint solves twice
    per_step = PICARD_PER_STEP * (51.0 + 55.0 * CYCLES_PER_PICARD)
    flops += csteps * per_step * (2.0 if kind == "adjoint" else 1.0)
    if kind == "adjoint":
        io += 8.0 * (case["modes"] * (case["nx"] * case["nz"] + 2 * case["samples"]) + case["samples"])
        flops += 4.0 * cells * case["modes"]
    return {"bytes": io, "flops": flops}


# ---------------------------------------------------------------- 64-bit restatement
M32 = 0xFFFFFFFF


def _philox(ctr, key):
    """Philox4x32-10 on int64 tensors holding 32-bit words."""
    c0, c1, c2, c3 = ctr
    k0, k1 = key
    for r in range(10):
        if r:
            k0, k1 = (k0 + 0x9E3779B9) & M32, (k1 + 0xBB67AE85) & M32

        def mul(m, c):                                  # 32 x 32 -> (high, low) without overflow
            lo = m * (c & 0xFFFF)
            hi = m * (c >> 16) + (lo >> 16)
            return hi >> 16, ((hi & 0xFFFF) << 16) | (lo & 0xFFFF)
        h0, l0 = mul(0xD2511F53, c0)
        h1, l1 = mul(0xCD9E8D57, c2)
        c0, c1, c2, c3 = h1 ^ c1 ^ k0, l1, h0 ^ c3 ^ k1, l0
    return c0, c1, c2, c3


def _noise(S, npts, seed, field):
    """Standard normals [S, npts] of one noise stream (level 0, samples 0 ... S-1)."""
    q = torch.arange(npts // 2, device="cuda", dtype=torch.int64)[None, :].expand(S, -1)
    s = torch.arange(S, device="cuda", dtype=torch.int64)[:, None].expand(-1, npts // 2)
    z = torch.zeros_like(q)
    c = _philox((q, z + field, s, z), (seed & M32, (seed >> 32) & M32))
    u = [(((a << 21) | (b >> 11)).double() + 0.5) * 2.0 ** -53 for a, b in ((c[0], c[1]), (c[2], c[3]))]
    r = torch.sqrt(-2.0 * torch.log(u[0]))
    return torch.stack((r * torch.cos(2 * math.pi * u[1]), r * torch.sin(2 * math.pi * u[1])), -1).reshape(S, npts)


def _covariance(m, px, pz, h):
    a = torch.arange(px, device="cuda", dtype=torch.float64)
    b = torch.arange(pz, device="cuda", dtype=torch.float64)
    a, b = torch.minimum(a, px - a) * h, torch.minimum(b, pz - b) * h
    r = torch.sqrt((a[None, :] / m.corr_len) ** 2 + (b[:, None] / (m.corr_len_z or m.corr_len)) ** 2)
    if m.nu == 0.0:
        return m.sigma2 * torch.exp(-r)
    if m.nu == 0.5:
        return m.sigma2 * torch.exp(-math.sqrt(2.0) * r)
    x = 2.0 * r                                         # nu = 1: x K_1(x)
    v = x * torch.special.modified_bessel_k1(torch.where(x > 0, x, torch.ones_like(x)))
    return m.sigma2 * torch.where(x > 0, v, torch.ones_like(v))


def _torus(m, nx, nz):
    px, pz = 2 * nx, 2 * nz
    for k in range(4):
        lam = torch.fft.fft2(_covariance(m, px, pz, 1.0 / nz)).real
        if float(lam.min() / lam.max()) >= -1e-12 or k == 3:
            return px, pz, torch.sqrt(lam.clamp_min(0.0))
        px, pz = 2 * px, 2 * pz


def _exact_fields(c, m, streams, pair):
    """Gaussian fields of the given noise streams: lists of [S, nz, nx] (and the
    coarse members by covariance upscaling)."""
    nx, nz, S = c["nx"], c["nz"], c["samples"]
    px, pz, sq = _torus(m, nx, nz)
    if pair:
        sqc = torch.sqrt(torch.fft.fft2(_covariance(m, px // 2, pz // 2, 2.0 / nz)).real.clamp_min(0.0))
    fine, coarse = [], []
    for f in streams:
        y = _noise(S, px * pz, m.seed, f).reshape(S, pz, px)
        fine.append(torch.fft.ifft2(sq * torch.fft.fft2(y)).real[:, :nz, :nx])
        if pair:
            yc = 0.5 * y.reshape(S, pz // 2, 2, px // 2, 2).sum((2, 4))
            coarse.append(torch.fft.ifft2(sqc * torch.fft.fft2(yc)).real[:, :nz // 2, :nx // 2])
    return fine, coarse


class _Steps:
    """Backward-Euler / modified Picard on the mixed form, cell-centred five-point
    finite volumes with harmonic-mean faces; linear solves by block elimination."""

    def __init__(self, pb, lnKs, alpha, n=None, ts=None, tr=None):
        self.pb, self.h = pb, 1.0 / pb.nz
        self.t2 = 2.0 / self.h ** 2
        self.Ks, self.a, self.n = torch.exp(lnKs), alpha, n
        self.ts = torch.full_like(alpha, pb.theta_s) if ts is None else ts
        self.tr = torch.full_like(alpha, pb.theta_r) if tr is None else tr
        self.Ttop = self.t2 * self.closure(torch.full_like(alpha, pb.p_top))[0][:, -1]
        self.Tbot = self.t2 * self.closure(torch.full_like(alpha, pb.p_bottom))[0][:, 0]

    def take(self, k):
        o = object.__new__(_Steps)
        o.pb, o.h, o.t2 = self.pb, self.h, self.t2
        for f in ("Ks", "a", "n", "ts", "tr", "Ttop", "Tbot"):
            v = getattr(self, f)
            setattr(o, f, None if v is None else v[k])
        return o

    def closure(self, p):
        """Conductivity, water content and capacity at head p."""
        dry = p < 0
        q = torch.where(dry, p, -torch.ones_like(p))
        if self.n is None:
            S = torch.exp(self.a * q)
            k, dS = S, self.a * S
        else:
            m = 1.0 - 1.0 / self.n
            an = (-self.a * q) ** self.n
            S = (1.0 + an) ** -m
            k = torch.sqrt(S) * (1.0 - (an / (1.0 + an)) ** m) ** 2
            dS = m * self.n * S * an / ((1.0 + an) * -q)
        one = torch.ones_like(p)
        return (self.Ks * torch.where(dry, k, one), self.tr + (self.ts - self.tr) * torch.where(dry, S, one),
                (self.ts - self.tr) * torch.where(dry, dS, 0 * one))

    def faces(self, K):
        return (self.t2 * K[:, :, :-1] * K[:, :, 1:] / (K[:, :, :-1] + K[:, :, 1:]),
                self.t2 * K[:, :-1] * K[:, 1:] / (K[:, :-1] + K[:, 1:]))

    def residual(self, p, K, th, th0):
        """(th - th0)/dt - div(K grad(p + z)) and the face coefficients."""
        tx, tz = self.faces(K)
        R_ = (th - th0) / self.pb.dt
        fx, fz = tx * (p[:, :, 1:] - p[:, :, :-1]), tz * (p[:, 1:] - p[:, :-1] + self.h)
        z = torch.zeros_like
        R_ = R_ - torch.cat((fx, z(fx[:, :, :1])), 2) + torch.cat((z(fx[:, :, :1]), fx), 2)
        top = self.Ttop * (self.pb.p_top - p[:, -1] + self.h / 2)
        bot = self.Tbot * (p[:, 0] - self.pb.p_bottom + self.h / 2)
        R_ = R_ - torch.cat((fz, top[:, None]), 1) + torch.cat((bot[:, None], fz), 1)
        return R_, tx, tz

    def diagonal(self, C, tx, tz):
        z = torch.zeros_like
        return (C / self.pb.dt + torch.cat((tx, z(C[:, :, :1])), 2) + torch.cat((z(C[:, :, :1]), tx), 2) +
                torch.cat((tz, self.Ttop[:, None]), 1) + torch.cat((self.Tbot[:, None], tz), 1))

    def step(self, p):
        """p^n -> p^(n+1) of every sample and whether its Picard iteration converged."""
        pb = self.pb
        S = p.shape[0]
        ok = torch.zeros(S, dtype=torch.bool, device=p.device)
        live = torch.arange(S, device=p.device)
        p = p.clone()
        th0 = self.closure(p)[1]
        for _ in range(pb.picard_maxit):
            me = self.take(live)
            q = p[live]
            K, th, C = me.closure(q)
            R_, tx, tz = me.residual(q, K, th, th0[live])
            d = _five_point_solve(me.diagonal(C, tx, tz), -tx, -tx, -tz, -tz, -R_)
            p[live] = q + d
            done = d.abs().amax((1, 2)) < pb.picard_tol
            ok[live[done]] = True
            live = live[~done]
            if live.numel() == 0:
                break
        return p, ok

    def initial(self):
        pb = self.pb
        if pb.init_decay > 0:
            z = (torch.arange(pb.nz, device="cuda", dtype=torch.float64) + 0.5) * self.h
            v = pb.p_init * (1.0 - torch.exp(-pb.init_decay * z))
            return v[None, :, None].expand_as(self.a).contiguous()
        return torch.full_like(self.a, pb.p_init)

    def qoi(self, p):
        K = self.Tbot / self.t2
        return (K * (2.0 * (p[:, 0] - self.pb.p_bottom) / self.h + 1.0)).mean(1)


def _five_point_solve(D, E, W, N, S, b):
    """Solve the five-point systems D x_P + E x_E + W x_W + N x_N + S x_S = b by
    block elimination over rows (E[k]: coefficient of cell k+1 in row k; W[k]: of
    cell k in row k+1; likewise N, S); rows run along the shorter side."""
    if D.shape[1] < D.shape[2]:
        t = lambda v: v.transpose(1, 2)  # noqa: E731
        return t(_five_point_solve(t(D), t(N), t(S), t(E), t(W), t(b)))
    nz = D.shape[1]
    inv, y = [], []
    for j in range(nz):
        A = torch.diag_embed(D[:, j]) + torch.diag_embed(E[:, j], 1) + torch.diag_embed(W[:, j], -1)
        r = b[:, j]
        if j:
            A = A - S[:, j - 1][:, :, None] * inv[-1] * N[:, j - 1][:, None, :]
            r = r - S[:, j - 1] * y[-1]
        inv.append(torch.linalg.inv_ex(A)[0])
        y.append((inv[-1] @ r[:, :, None])[:, :, 0])
    x = [y[-1]]
    for j in range(nz - 2, -1, -1):
        x.append(y[j] - (inv[j] @ (N[:, j] * x[-1])[:, :, None])[:, :, 0])
    return torch.stack(x[::-1], 1)


def _exact_solve(c, d):
    o = _Steps(_problem(c), d["lnKs"], d["alpha"] * c.get("scale", 1.0), d.get("n"), d.get("theta_s"),
               d.get("theta_r"))
    p = o.initial()
    ok = torch.ones(p.shape[0], dtype=torch.bool, device="cuda")
    for _ in range(c["steps"]):
        k = torch.nonzero(ok)[:, 0]
        if k.numel() == 0:
            break
        p[k], ok[k] = o.take(k).step(p[k])
    p = p.masked_fill(~ok[:, None, None], math.nan)
    return o.qoi(p), p


def _exact_adjoint(c, d):
    """QoI and its gradient by the adjoint of the converged steps."""
    lk = torch.einsum("sj,jzx->szx", d["xi"], d["basis"])
    o = _Steps(_problem(c), lk, d["alpha"])
    ps, ok = [o.initial()], torch.ones(lk.shape[0], dtype=torch.bool, device="cuda")
    for _ in range(c["steps"]):
        p, good = o.step(ps[-1])
        ok &= good
        ps.append(p)
    m = lk.clone().requires_grad_(True)
    om = _Steps(_problem(c), m, d["alpha"])
    total = om.qoi(ps[-1]).sum()
    lam = None
    h = o.h
    for k in range(c["steps"], 0, -1):
        p = ps[k]
        K, th, C = o.closure(p)
        if lam is None:
            rhs = torch.zeros_like(p)
            rhs[:, 0] = o.Tbot / o.t2 * (2.0 / h) / p.shape[2]
        else:
            rhs = C / o.pb.dt * lam
        dK = torch.where(p < 0, o.a * K, torch.zeros_like(K))
        tx, tz = o.faces(K)
        gx, gz = p[:, :, 1:] - p[:, :, :-1], p[:, 1:] - p[:, :-1] + h
        sx, sz = o.t2 / (K[:, :, 1:] + K[:, :, :-1]) ** 2, o.t2 / (K[:, 1:] + K[:, :-1]) ** 2
        e = tx - gx * sx * K[:, :, 1:] ** 2 * dK[:, :, :-1]           # -dR_east/dp_cell, and so on
        w = tx + gx * sx * K[:, :, :-1] ** 2 * dK[:, :, 1:]
        n = tz - gz * sz * K[:, 1:] ** 2 * dK[:, :-1]
        s = tz + gz * sz * K[:, :-1] ** 2 * dK[:, 1:]
        z = torch.zeros_like
        D = (C / o.pb.dt + torch.cat((e, z(p[:, :, :1])), 2) + torch.cat((z(p[:, :, :1]), w), 2) +
             torch.cat((n, o.Ttop[:, None]), 1) + torch.cat((o.Tbot[:, None], s), 1))
        lam = _five_point_solve(D, -e, -w, -n, -s, rhs)
        Km, thm, _ = om.closure(p)
        total = total - (lam * om.residual(p, Km, thm, om.closure(ps[k - 1])[1])[0]).sum()
    g = torch.autograd.grad(total, m)[0]
    dq = torch.einsum("jzx,szx->sj", d["basis"], g)
    return (o.qoi(ps[-1]).masked_fill(~ok, math.nan), dq.masked_fill(~ok[:, None], math.nan))


def exact(case, seed):
    kind, c = case["kind"], case
    if kind == "mlmc":
        return None
    if kind == "fields":
        m = _model(c, seed)
        (a, b), _ = _exact_fields(c, m, (0, 1), False)
        return a.contiguous(), m.alpha_lo + m.alpha_span * _phi(b)
    if kind == "soil_pair":
        m, s = R.soil_field_model(3.0, _model(c, seed)), R.SoilModel()
        lo = (0.0, m.alpha_lo, s.n_bl - s.d_n, s.theta_s_bl - s.d_theta_s, s.theta_r_bl - s.d_theta_r)
        span = (0.0, m.alpha_span, 2 * s.d_n, 2 * s.d_theta_s, 2 * s.d_theta_r)
        both = _exact_fields(c, m, (0, 1, 2, 3, 4), True)
        return tuple(tuple(math.log(s.ks_bl) + z if k == 0 else lo[k] + span[k] * _phi(z) for k, z in enumerate(side))
                     for side in both)
    # the direct solves cost about side^2 work a cell and a launch or ten a row: small batches only
    short = min(c["nx"], c["nz"])
    if c["nx"] * c["nz"] * c["samples"] * c["steps"] * short ** 2 > 2e10 or max(c["nx"], c["nz"]) * c["steps"] > 700:
        return None
    d = _inputs(c, seed)
    if kind == "adjoint":
        return _exact_adjoint(c, d)
    qoi, p = _exact_solve(c, d)
    return qoi, p, None
