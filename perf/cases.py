"""The calls this library is measured on: what a program that estimates flow
through random media has it do, through the Python binding, and how large.

Every case is one public call (or the training and the estimate of one
estimator run).  Kinds:

  level      points -> KL field -> FMG solves -> level sums of one MLMC level
             (mlmc_sample_level), FP64 or mixed, MC or randomized Sobol'
  solve      FMG solves of fields the caller has (fmg_solve_batch)
  uneven     groups of different grids as one batch (fmg_solve_uneven)
  field      KL field synthesis alone (kl_field_batch)
  surrogate  evaluation of the surrogate network on MC samples
  train      training of the surrogate network
  estimate   the whole multilevel estimate (mlmc_estimate)

The random fields have the exponential covariance of the method: the modes are
the plane waves of a periodic box around the unit square (a cosine and a sine
each, so the variance is the same everywhere) with the spectral density of
that covariance, the M largest kept.
"""
import math

import numpy as np
import torch

import paper_1910_04727_gb300 as fm

DEV = "cuda"
TOL, QTOL = 1e-12, 1e-10     # stopping rule of the converged forms (as the benchmark's)
MIXED_CYCLES = 6             # FP32 V-cycles per FP64 residual of the mixed form
FORMS = ("fp64_fixed", "fp64_converged", "mixed")
PERIOD = 1.5                 # side of the periodic box
GRIDS = (16, 32, 64, 128, 256)
MC_STREAM = 1                # purpose word of the Philox streams of MC points
S_STREAM = 12                # Philox stream of the surrogate level's samples

# Most samples of a drawn level, solve or group, by form and grid: at most
# some 50 ms of work at the rates of a GB300.
MOST = {
    "fp64_fixed": {16: 60000, 32: 20000, 64: 8000, 128: 2000, 256: 700, 512: 150, 1024: 30},
    "fp64_converged": {16: 20000, 32: 7000, 64: 2500, 128: 600, 256: 200, 512: 40, 1024: 8},
    "mixed": {16: 60000, 32: 15000, 64: 4000, 128: 1200, 256: 600, 512: 150, 1024: 30},
}


def listed():
    return [
        # one level alone, the smallest estimator in use: 256 samples of 32 x 32
        {"name": "level32_fp64", "kind": "level", "form": "fp64_fixed", "n": 32, "modes": 64, "samples": 256,
         "sampler": "mc"},
        # the method's own fixed FP64 schedule on a middle level of five
        {"name": "level64_fp64", "kind": "level", "form": "fp64_fixed", "n": 64, "modes": 128, "samples": 5304,
         "sampler": "mc"},
        # FP64 to a tolerance: the reference results of a study
        {"name": "level128_fp64conv", "kind": "level", "form": "fp64_converged", "n": 128, "modes": 128,
         "samples": 401, "sampler": "mc"},
        # the bulk of the samples: level 0 in the mixed form, randomized QMC
        {"name": "level16_mixed", "kind": "level", "form": "mixed", "n": 16, "modes": 128, "samples": 47001,
         "sampler": "sobol"},
        # the pilot run of the finest of five levels
        {"name": "level256_mixed", "kind": "level", "form": "mixed", "n": 256, "modes": 128, "samples": 1000,
         "sampler": "mc"},
        # a few large, rough fields of the caller's, with the robust step and the pressure returned
        {"name": "solve1024_mixed", "kind": "solve", "form": "mixed", "n": 1024, "samples": 7, "sigma2": 2.0,
         "lam": 0.1, "energy": True, "bc_case": 2, "pressure": True},
        # batches of a shared cluster job: all grids at once
        {"name": "uneven_mixed", "kind": "uneven", "form": "mixed", "n": 64, "groups": 4, "samples": 1537},
        # field synthesis where FP64 is asked for
        {"name": "field64_fp64", "kind": "field", "form": "fp64", "n": 64, "modes": 128, "samples": 2000},
        # field synthesis of the mixed form, many modes on a fine grid
        {"name": "field256_bf16x3", "kind": "field", "form": "bf16x3", "n": 256, "modes": 256, "samples": 500},
        # the surrogate level of an estimate
        {"name": "surrogate_1m", "kind": "surrogate", "modes": 128, "samples": 1000003},
        # training of the surrogate, inside every estimate that uses it
        {"name": "train_20480", "kind": "train", "modes": 128, "pairs": 20480, "epochs": 20, "batch": 1024},
        # the whole estimate: five levels, surrogate trained beside the pilot round
        {"name": "estimate5", "kind": "estimate", "levels": 5, "modes": 128, "eps": 1e-3, "qmc": False,
         "surrogate": True},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("level", "level", "level", "solve", "solve", "uneven", "field", "field", "surrogate", "train",
                       "estimate"))
    if kind == "level":
        form, n = rng.choice(FORMS), rng.choice(GRIDS)
        return {"kind": kind, "form": form, "n": n, "modes": _log_int(rng, 20, 300),
                "samples": _log_int(rng, 16, MOST[form][n]), "sampler": rng.choice(("mc", "mc", "sobol", "owen"))}
    if kind == "solve":
        form, n = rng.choice(FORMS), rng.choice((32, 64, 128, 256, 512, 1024))
        energy = form != "fp64_fixed" and rng.random() < 0.3
        most = max(1, MOST[form][n] // (4 if energy else 1))
        return {"kind": kind, "form": form, "n": n, "samples": _log_int(rng, 1, most),
                "sigma2": round(rng.uniform(0.5, 2.0 if energy else 1.0), 2), "lam": round(rng.uniform(0.1, 0.5), 2),
                "energy": energy, "bc_case": rng.choice((1, 2, 2)), "pressure": rng.random() < 0.5}
    if kind == "uneven":
        form, n, groups = rng.choice(("mixed", "mixed", "fp64_fixed")), rng.choice((16, 32, 64)), rng.randint(2, 4)
        return {"kind": kind, "form": form, "n": n, "groups": groups,
                "samples": _log_int(rng, 64, min(MOST[form][n] // 2, 2500))}
    if kind == "field":
        form, n, modes = rng.choice(("fp64", "bf16x3")), rng.choice(GRIDS), _log_int(rng, 16, 600)
        most = min(2e10 / (n * n * modes) if form == "fp64" else 1e8 / (n * n), 60000)
        return {"kind": kind, "form": form, "n": n, "modes": modes, "samples": _log_int(rng, 8, max(8, most))}
    if kind == "surrogate":
        return {"kind": kind, "modes": _log_int(rng, 16, 256), "samples": _log_int(rng, 1000, 3000000)}
    if kind == "train":
        batch = rng.choice((256, 512, 1024, 2048))
        pairs = max(batch, _log_int(rng, 2048, 24000))
        return {"kind": kind, "modes": _log_int(rng, 32, 200), "pairs": pairs,
                "epochs": max(1, min(rng.randint(8, 20), 400 * batch // pairs)), "batch": batch}
    surrogate = rng.random() < 0.7
    return {"kind": kind, "levels": rng.randint(2, 5), "modes": _log_int(rng, 48, 160),
            "eps": round(math.exp(rng.uniform(math.log(1.5e-3 if surrogate else 4e-3), math.log(1e-2))), 5),
            "qmc": rng.random() < 0.5, "surrogate": surrogate}


# ------------------------------------------------------------------ inputs
def _generator(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 7919 + 17)
    return g


def _basis(n, modes, sigma2=1.0, lam=0.3):
    """[n^2][modes] sqrt(theta_k) phi_k at the cell centres of the grid."""
    top = int(math.isqrt(modes)) + 4
    kx, ky = np.meshgrid(np.arange(-top, top + 1), np.arange(0, top + 1), indexing="ij")
    kx, ky = kx.ravel(), ky.ravel()
    half = (ky > 0) | (kx > 0)                  # one of each pair k, -k, and the constant apart
    kx, ky = np.append(kx[half], 0), np.append(ky[half], 0)

    def density(k2):
        return (1.0 / lam ** 2 + (2 * np.pi / PERIOD) ** 2 * k2) ** -1.5
    i = np.arange(-300.0, 301.0)
    total = density(i[:, None] ** 2 + i[None, :] ** 2).sum()
    order = np.argsort(-density(kx ** 2 + ky ** 2), kind="stable")
    pick, odd = [], []
    for k in order:                             # a cosine and a sine for every wave vector
        for sine in ((0,) if kx[k] == ky[k] == 0 else (0, 1)):
            pick.append(k)
            odd.append(sine)
    pick, odd = np.array(pick[:modes]), np.array(odd[:modes])
    theta = density(kx[pick] ** 2 + ky[pick] ** 2) * np.where((kx[pick] == 0) & (ky[pick] == 0), 1.0, 2.0)
    x = (torch.arange(n, dtype=torch.float64, device=DEV) + 0.5) / n
    w = 2 * math.pi / PERIOD
    px = x[None, :, None] * (w * torch.tensor(kx[pick], dtype=torch.float64, device=DEV))
    py = x[:, None, None] * (w * torch.tensor(ky[pick], dtype=torch.float64, device=DEV))
    amp = torch.tensor(np.sqrt(sigma2 * theta / total), device=DEV)
    shift = torch.tensor(odd * (math.pi / 2), device=DEV)
    return (torch.cos(px + py - shift) * amp).reshape(n * n, modes).contiguous()


def _fields(n, samples, sigma2, lam, seed, modes=256):
    xi = torch.randn((samples, modes), generator=_generator(seed), dtype=torch.float64, device=DEV)
    return torch.exp(xi @ _basis(n, modes, sigma2, lam).T).reshape(samples, n, n).contiguous()


def _form(form):
    return dict(precision=fm.FM_PREC_MIXED if form == "mixed" else fm.FM_PREC_FP64, converged=form != "fp64_fixed",
                tol=TOL, qtol=QTOL, max_cycles=300, ir_cycles=MIXED_CYCLES if form == "mixed" else 0)


def _group_sizes(case):
    """Grids n, 2n, 4n, ... with a quarter of the samples from each to the next."""
    grids = [case["n"] << g for g in range(case["groups"])]
    w = [4.0 ** -g for g in range(case["groups"])]
    return [(n, max(1, int(case["samples"] * v / sum(w)))) for n, v in zip(grids, w)]


def prepare(case, seed):
    kind = case["kind"]
    if kind == "level":
        n = case["n"]
        levels = max(1, int(math.log2(n // 16)) + 1) if n > 32 else 1
        ctx = fm.Context(levels, n >> (levels - 1), case["modes"], seed=seed, **_form(case["form"]),
                         qmc_rule=1 if case["sampler"] == "owen" else 0)
        ctx.kl_basis_set(_basis(n, case["modes"]))
        return {"case": case, "ctx": ctx, "level": levels - 1, "shift": -1 if case["sampler"] == "mc" else 3}
    if kind == "solve":
        ctx = fm.Context(1, case["n"], 8, bc_case=case["bc_case"], pS=0.3, pN=0.6, energy_step=case["energy"],
                         **_form(case["form"]))
        return {"case": case, "ctx": ctx, "K": _fields(case["n"], case["samples"], case["sigma2"], case["lam"], seed)}
    if kind == "uneven":
        ctx = fm.Context(1, case["n"], 8, **_form(case["form"]))
        return {"case": case, "ctx": ctx,
                "K": [_fields(n, s, 1.0, 0.3, seed + 31 * n) for n, s in _group_sizes(case)]}
    if kind == "field":
        ctx = fm.Context(1, case["n"], case["modes"], kl_mode=1 if case["form"] == "fp64" else 3)
        ctx.kl_basis_set(_basis(case["n"], case["modes"]))
        xi = torch.randn((case["samples"], case["modes"]), generator=_generator(seed), dtype=torch.float64, device=DEV)
        return {"case": case, "ctx": ctx, "xi": xi}
    if kind == "surrogate":
        ctx = fm.Context(1, 16, case["modes"], seed=seed)
        r = np.random.default_rng(seed)
        m = case["modes"]
        parts = []
        for rows, fan in ((256, m), (256, 256), (256, 256), (1, 256)):
            a = 1.0 / math.sqrt(fan)
            parts += [r.uniform(-a, a, rows * fan) * 1.7, r.uniform(-a, a, rows)]
        params = np.concatenate(parts).astype(np.float32)
        ctx.surrogate_set_params(params, mu=1.1, sd=0.4)
        return {"case": case, "ctx": ctx, "params": params}
    if kind == "train":
        ctx = fm.Context(1, 16, case["modes"], seed=seed, **_form("mixed"))
        ctx.kl_basis_set(_basis(16, case["modes"]))
        return {"case": case, "ctx": ctx, "seed": seed}
    n = 16 << (case["levels"] - 1)
    ctx = fm.Context(case["levels"], 16, case["modes"], seed=seed, n_shifts=16, **_form("mixed"))
    ctx.kl_basis_set(_basis(n, case["modes"]))
    return {"case": case, "ctx": ctx, "seed": seed}


# ------------------------------------------------------------------ the calls
def run(state):
    case, ctx = state["case"], state["ctx"]
    kind = case["kind"]
    if kind == "level":
        sums = ctx.new_sums()
        qf, qc = ctx.mlmc_sample_level(state["level"], 0, case["samples"], state["shift"], sums=sums[0], want_q=True)
        return {"qf": qf, "qc": qc, "sums": sums}
    if kind == "solve":
        qf, qc, p = ctx.fmg_solve_batch(state["K"], want_p=case["pressure"])
        return {"qf": qf, "qc": qc, "p": p}
    if kind == "uneven":
        return [(qf, qc) for qf, qc, _ in ctx.solve_uneven(state["K"])]
    if kind == "field":
        return {"K": ctx.kl_field_batch(0, state["xi"])}
    if kind == "surrogate":
        return {"s": ctx.surrogate_eval_mc(S_STREAM, 0, case["samples"])}
    if kind == "train":
        r = ctx.surrogate_train(n_train=case["pairs"], epochs=case["epochs"], lr=4e-3, seed=state["seed"] & 0xffff,
                                batch=case["batch"], target_tol=1e-6)
        return {"params": ctx.surrogate_get_params(),
                "report": [r["loss_first"], r["loss_last"], r["mu"], r["sd"], r["corr"], r["var_residual"]]}
    if case["surrogate"]:
        ctx.surrogate_train(n_train=20480, epochs=20, lr=4e-3, seed=state["seed"] & 0xffff, batch=1024,
                            target_tol=1e-6, async_run=True)
    r = ctx.mlmc_estimate(case["eps"], qmc=case["qmc"], n_pilot=32 if case["qmc"] else 1000,
                          surrogate=case["surrogate"], surrogate_cost=0.027, batched=True)
    if case["surrogate"]:
        ctx.surrogate_train_finish()
    return {k: np.asarray(r[k]) for k in ("estimate", "var_estimator", "means", "V", "N", "mean_s", "var_s", "N_s",
                                          "rounds")}


# ------------------------------------------------------------------ work
def _solve_work(case, n, samples):
    """Full multigrid of `samples` n x n problems.  Fixed schedule: nu0 = 2 V(2,2) cycles per stage.
    Converged: 12 cycles on each of the two finest stages, which a contraction of 0.1 needs for TOL."""
    cycles, stages = (2, [1.0, 0.25, 0.0625]) if case["form"] == "fp64_fixed" else (12, [1.0, 0.25])
    per_cell = 4 / 3 * (4 * 10 + 18)          # four sweeps, residual, transfers, on a grid and below it
    cells = float(samples) * n * n
    return {"bytes": cells * 8 + 16.0 * samples, "flops": sum(stages) * cycles * per_cell * cells}


def _add(*parts):
    return {k: float(sum(p[k] for p in parts)) for k in ("bytes", "flops")}


def _network_flops(m):
    return 2.0 * (m * 256 + 2 * 256 * 256 + 256)


def work(case):
    kind = case["kind"]
    if kind == "level":
        n, s, m = case["n"], case["samples"], case["modes"]
        w = _solve_work(case, n, s)
        return {"bytes": 8.0 * n * n * m + 16.0 * s, "flops": w["flops"] + 2.0 * n * n * m * s}
    if kind == "solve":
        w = _solve_work(case, case["n"], case["samples"])
        return _add(w, {"bytes": 8.0 * case["samples"] * case["n"] ** 2 if case["pressure"] else 0.0, "flops": 0.0})
    if kind == "uneven":
        return _add(*[_solve_work(case, n, s) for n, s in _group_sizes(case)])
    if kind == "field":
        n2, s, m = case["n"] ** 2, case["samples"], case["modes"]
        return {"bytes": 8.0 * (n2 * m + s * m + n2 * s), "flops": 2.0 * n2 * m * s}
    if kind == "surrogate":
        return {"bytes": 8.0 * case["samples"], "flops": case["samples"] * _network_flops(case["modes"])}
    if kind == "train":
        steps = case["pairs"] // case["batch"] * case["epochs"]
        mixed = {"form": "mixed"}
        return _add(_solve_work(mixed, 16, case["pairs"]),
                    {"bytes": 8.0 * case["pairs"] * case["modes"],
                     "flops": 3.0 * steps * case["batch"] * _network_flops(case["modes"])})
    # an estimate: at least the pilot samples of every level
    pilot = 32 * 16 if case["qmc"] else 1000
    parts = [_solve_work({"form": "mixed"}, 16 << l, pilot) for l in range(case["levels"])]
    if case["surrogate"]:
        parts.append(_solve_work({"form": "mixed"}, 16, 20480))
        parts.append({"bytes": 0.0, "flops": 3.0 * 400 * 1024 * _network_flops(case["modes"])})
    return _add(*parts)


# ------------------------------------------------------------------ 64-bit results in plain torch
_M0, _M1 = 0xD2E7470EE14C6C93, 0xCA5A826395121157
_W0, _W1 = 0x9E3779B97F4A7C15, 0xBB67AE8584CAA73B


def _mulhilo(a, b):
    mask = np.uint64(0xFFFFFFFF)
    a0, a1 = np.uint64(a & 0xFFFFFFFF), np.uint64(a >> 32)
    b0, b1 = b & mask, b >> np.uint64(32)
    mid = a1 * b0 + ((a0 * b0) >> np.uint64(32))
    mid2 = a0 * b1 + (mid & mask)
    return a1 * b1 + (mid >> np.uint64(32)) + (mid2 >> np.uint64(32)), np.uint64(a) * b


def _philox_words(seed, stream, samples, dim):
    """Words [samples][dim] of Philox4x64-10 (Salmon et al. 2011), counter (k / 4, sample, 0, 0)."""
    groups = (dim + 3) // 4
    with np.errstate(over="ignore"):
        c = [np.broadcast_to(np.arange(groups, dtype=np.uint64), (samples, groups)).copy(),
             np.broadcast_to(np.arange(samples, dtype=np.uint64)[:, None], (samples, groups)).copy(),
             np.zeros((samples, groups), np.uint64), np.zeros((samples, groups), np.uint64)]
        k0, k1 = int(seed), (MC_STREAM << 32) | int(stream)
        for _ in range(10):
            h0, l0 = _mulhilo(_M0, c[0])
            h1, l1 = _mulhilo(_M1, c[2])
            c = [h1 ^ c[1] ^ np.uint64(k0), l1, h0 ^ c[3] ^ np.uint64(k1), l0]
            k0, k1 = (k0 + _W0) & (2 ** 64 - 1), (k1 + _W1) & (2 ** 64 - 1)
    return np.stack(c, axis=-1).reshape(samples, 4 * groups)[:, :dim]


def _normals(seed, stream, samples, dim):
    u = ((_philox_words(seed, stream, samples, dim) >> np.uint64(11)).astype(np.float64) + 0.5) * 2.0 ** -53
    return torch.special.ndtri(torch.from_numpy(u).to(DEV))


class _Grid:
    """The finite-volume operator of one coefficient field [S][n][n] (Dirichlet west / east, and south / north with
    ns), red-black Gauss-Seidel and residual."""

    def __init__(self, K, ns):
        self.n, self.ns, self.K = K.shape[-1], ns, K
        z = torch.zeros_like(K)
        te, tn = z.clone(), z.clone()
        te[:, :, :-1] = 2 * K[:, :, :-1] * K[:, :, 1:] / (K[:, :, :-1] + K[:, :, 1:])
        tn[:, :-1, :] = 2 * K[:, :-1, :] * K[:, 1:, :] / (K[:, :-1, :] + K[:, 1:, :])
        self.te, self.tn = te, tn
        D = te + tn
        D[:, :, 1:] += te[:, :, :-1]
        D[:, 1:, :] += tn[:, :-1, :]
        D[:, :, 0] += 2 * K[:, :, 0]
        D[:, :, -1] += 2 * K[:, :, -1]
        if ns:
            D[:, 0, :] += 2 * K[:, 0, :]
            D[:, -1, :] += 2 * K[:, -1, :]
        self.D = D
        i = torch.arange(self.n, device=K.device)
        self.red = ((i[:, None] + i[None, :]) % 2 == 0)

    def off(self, p):
        v = torch.zeros_like(p)
        fe, fn = self.te[:, :, :-1], self.tn[:, :-1, :]
        v[:, :, 1:] += fe * p[:, :, :-1]
        v[:, :, :-1] += fe * p[:, :, 1:]
        v[:, 1:, :] += fn * p[:, :-1, :]
        v[:, :-1, :] += fn * p[:, 1:, :]
        return v

    def apply(self, p):
        return self.D * p - self.off(p)

    def sweep(self, p, b):
        p = torch.where(self.red, (b + self.off(p)) / self.D, p)
        return torch.where(self.red, p, (b + self.off(p)) / self.D)

    def dense_solve(self, b):
        m = self.n * self.n
        e = torch.eye(m, dtype=b.dtype, device=b.device).reshape(m, 1, self.n, self.n)
        A = torch.stack([self.apply(e[k].expand_as(self.D)).reshape(-1, m) for k in range(m)], dim=-1)
        return torch.linalg.solve(A, b.reshape(-1, m, 1)).reshape(b.shape)


def _prolong(u, g, ns):
    """Bilinear cell-centred interpolation with ghosts 2g - u across Dirichlet edges g = (w, e, s, n)."""
    u = torch.cat([2 * g[0] - u[:, :, :1], u, 2 * g[1] - u[:, :, -1:]], dim=2)
    lo, hi = u[:, :1], u[:, -1:]
    u = torch.cat([2 * g[2] - lo if ns else lo, u, 2 * g[3] - hi if ns else hi], dim=1)
    own, out = u[:, 1:-1, 1:-1], []
    for dy in (0, 2):
        row = []
        for dx in (0, 2):
            ny, nx = u[:, dy:u.shape[1] - 2 + dy], u[:, 1:-1]
            row.append((9 * own + 3 * nx[:, :, dx:u.shape[2] - 2 + dx] + 3 * ny[:, :, 1:-1]
                        + ny[:, :, dx:u.shape[2] - 2 + dx]) / 16)
        out.append(torch.stack(row, dim=-1).flatten(-2))
    return torch.stack(out, dim=2).flatten(1, 2)


def _fmg(K, fixed, bnd, ns):
    """(qf, qc, p): full multigrid on fields K [S][n][n], two V(2,2) cycles per stage, or (not fixed) the two finest
    stages to rounding level by energy-minimising corrections."""
    m = int(math.log2(K.shape[-1] // 4))
    Ks = [K]
    for _ in range(m):
        Ks.insert(0, Ks[0][:, ::2, ::2].contiguous())
    stage = [_Grid(k, ns) for k in Ks]

    def geo(k):
        return torch.exp(0.25 * sum(torch.log(k[:, a::2, b::2]) for a in (0, 1) for b in (0, 1)))
    corr = [_Grid(geo(k), ns) for k in Ks[1:]]
    zero = (0.0, 0.0, 0.0, 0.0)

    def cycle(k, G, p, b, step):
        if k == 0:
            return G.dense_solve(b)
        for _ in range(2):
            p = G.sweep(p, b)
        r = b - G.apply(p)
        rc = r[:, ::2, ::2] + r[:, ::2, 1::2] + r[:, 1::2, ::2] + r[:, 1::2, 1::2]
        d = _prolong(cycle(k - 1, corr[k - 1], torch.zeros_like(rc), rc, step), zero, ns)
        if step:
            alpha = (r * d).sum((1, 2)) / (d * G.apply(d)).sum((1, 2)).clamp_min(1e-300)
            d = d * alpha[:, None, None]
        p = p + d
        for _ in range(2):
            p = G.sweep(p, b)
        return p

    def qoi(G, p):
        if ns:
            h = G.n // 2
            return p[:, h - 1:h + 1, h - 1:h + 1].mean((1, 2))
        return (2 * G.K[:, :, -1] * (p[:, :, -1] - bnd[1])).sum(1)
    p, qc = None, None
    for k in range(m + 1):
        G = stage[k]
        b = torch.zeros_like(G.K)
        b[:, :, 0] += 2 * G.K[:, :, 0] * bnd[0]
        b[:, :, -1] += 2 * G.K[:, :, -1] * bnd[1]
        if ns:
            b[:, 0, :] += 2 * G.K[:, 0, :] * bnd[2]
            b[:, -1, :] += 2 * G.K[:, -1, :] * bnd[3]
        if k == 0:
            p = G.dense_solve(b)
        else:
            p = _prolong(p, bnd, ns)
            if fixed or k < m - 1:
                for _ in range(2):
                    p = cycle(k, G, p, b, False)
            else:
                last = math.inf
                for it in range(120):
                    r = float(((b - G.apply(p)).square().sum((1, 2)) / b.square().sum((1, 2))).max().sqrt())
                    if r < 2e-15 or (r < 1e-13 and r > 0.7 * last):
                        break
                    last, p = r, cycle(k, G, p, b, True)
        if k == m - 1:
            qc = qoi(G, p)
    return qoi(stage[m], p), qc, p


def _fmg_in_parts(K, fixed, bnd=(1.0, 0.0, 0.0, 0.0), ns=False, pressure=False):
    most = max(1, (24 << 20) // K.shape[-1] ** 2)
    parts = [_fmg(K[i:i + most], fixed, bnd, ns) for i in range(0, K.shape[0], most)]
    return (torch.cat([p[0] for p in parts]), torch.cat([p[1] for p in parts]),
            torch.cat([p[2] for p in parts]) if pressure else None)


def exact(case, seed):
    kind = case["kind"]
    if kind == "level":
        if case["sampler"] != "mc":
            return None
        levels = max(1, int(math.log2(case["n"] // 16)) + 1) if case["n"] > 32 else 1
        xi = _normals(seed, levels - 1, case["samples"], case["modes"])
        K = torch.exp(xi @ _basis(case["n"], case["modes"]).T).reshape(-1, case["n"], case["n"])
        qf, qc, _ = _fmg_in_parts(K, case["form"] == "fp64_fixed")
        return {"qf": qf, "qc": qc, "sums": None}
    if kind == "solve":
        K = _fields(case["n"], case["samples"], case["sigma2"], case["lam"], seed)
        ns = case["bc_case"] == 1
        qf, qc, p = _fmg_in_parts(K, case["form"] == "fp64_fixed", (1.0, 0.0, 0.3, 0.6), ns, case["pressure"])
        return {"qf": qf, "qc": qc, "p": p}
    if kind == "uneven":
        return [_fmg_in_parts(_fields(n, s, 1.0, 0.3, seed + 31 * n), case["form"] == "fp64_fixed")[:2]
                for n, s in _group_sizes(case)]
    if kind == "field":
        xi = torch.randn((case["samples"], case["modes"]), generator=_generator(seed), dtype=torch.float64, device=DEV)
        K = torch.exp(xi @ _basis(case["n"], case["modes"]).T)
        return {"K": K.reshape(-1, case["n"], case["n"])}
    if kind == "surrogate":
        if case["samples"] * case["modes"] > 140e6:
            return None
        s = prepare(case, seed)
        w = _philox_words(seed, S_STREAM, case["samples"], case["modes"])
        x = torch.special.ndtri(torch.from_numpy(((w >> np.uint64(41)).astype(np.float64) + 0.5) * 2.0 ** -23).to(DEV))
        o, m = 0, case["modes"]
        P = torch.from_numpy(s["params"]).to(DEV, torch.float64)
        for rows, fan in ((256, m), (256, 256), (256, 256), (1, 256)):
            W, bias = P[o:o + rows * fan].reshape(rows, fan), P[o + rows * fan:o + rows * fan + rows]
            x, o = x @ W.T + bias, o + rows * fan + rows
            if rows > 1:
                x = torch.nn.functional.gelu(x)
        return {"s": 1.1 + 0.4 * x[:, 0]}
    return None   # a training run or an estimate: thousands of dependent steps
