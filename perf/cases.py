"""Performance cases: the calls that a user of the package makes, over the sizes they are made at.

A case is one of
  step     one evaluation of the particle model: seed, n_steps of the time step, deposition tally
           (single samples in FP64, batches in MIXED, all-stick and rebound, with and without
           particle-particle contact, ragged sample sizes);
  p3m      the same with P3M electrostatics for one large sample;
  adjoint  value and gradient of the smoothed V_dep+ through the autograd function;
  lf       the 1-D Eulerian low-fidelity model on a table of samples;
  mfmc     the two-model MFMC Sobol' estimators with bootstrap intervals.

exact() restates each of them in 64 bits with torch and numpy alone.
"""
import math

import numpy as np
import torch
import torch.utils.checkpoint

from paper_2205_04979_gb300 import pdq

DEV = "cuda"
R_PLUS, L_PLUS = 180.0, 720.0
GRIDS = {"small": (64, 32, 64), "large": (128, 64, 128)}
PRECISION = {"fp64": pdq.FP64, "mixed": pdq.MIXED}
MODES = {"stick": pdq.STICK, "rebound": pdq.REBOUND}


def st_classes(n):
    """The size classes of an n-class study: St+ = 10 alone, else log-spaced 0.1..10 (10 classes: 0.1..100)."""
    if n == 1:
        return [10.0]
    return [float(v) for v in np.geomspace(0.1, 100.0 if n >= 10 else 10.0, n)]


def step_case(name, precision, samples, lo, hi, classes, steps, grid="small", dt=0.05, sigma=0.0, mode="stick",
              contact=False, neg=0.0, compact=100, block=-1, variant=0):
    """block -1: the autotuner's choice; otherwise the given threads per CTA and pair variant."""
    c = dict(kind="step", precision=precision, samples=samples, lo=lo, hi=hi, classes=classes, steps=steps, grid=grid,
             dt=dt, sigma=sigma, mode=mode, contact=contact, neg=neg, compact=compact, block=block, variant=variant)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest run: one sample of 1,000 particles in FP64, bound by latency and the FP64 pipe
        step_case("fp64_single", "fp64", 1, 1000, 1000, 1, 40, dt=0.1, compact=0),
        # the paper's scale in FP64 by direct summation: 10 classes, lognormal charges; a long run
        # keeps the launch configuration that it tuned once
        step_case("fp64_paper_scale", "fp64", 1, 100_000, 100_000, 10, 2, grid="large", sigma=0.5, compact=0, block=64,
                  variant=3),
        # V_dep+ of a handful of inputs: 16 samples of 4,096 particles (the accuracy study's size)
        step_case("mixed_vdep_16", "mixed", 16, 4096, 4096, 5, 10),
        # a Sobol' study of the capture efficiency: 64 pick-freeze groups of 5 runs, rebound walls
        step_case("mixed_sobol_rebound", "mixed", 320, 4096, 4096, 3, 4, mode="rebound"),
        # the batched study: 1,024 samples of 4,096 to 32,768 particles
        step_case("mixed_batch_1024", "mixed", 1024, 4096, 32768, 5, 2, grid="large", block=128, variant=3),
        # charges of both signs with collisions and van der Waals forces between particles
        step_case("mixed_contact", "mixed", 48, 4096, 16384, 5, 2, grid="large", contact=True, neg=0.5),
        # gradient of a few samples, as an optimiser or a check against differences asks for it
        dict(name="adjoint_16", kind="adjoint", precision="mixed", samples=16, count=2048, classes=3, steps=20, ckpt=10,
             eps=0.5, store=False, mode="stick"),
        # gradients for the sensitivity bounds: 256 samples of 16,384 particles, pair sums kept
        dict(name="adjoint_256", kind="adjoint", precision="mixed", samples=256, count=16384, classes=3, steps=4, ckpt=2,
             eps=0.1, store=True, mode="stick"),
        # the paper's electrostatics: one sample of a million particles
        dict(name="p3m_1m", kind="p3m", count=1_000_000, classes=10, steps=2, mesh=123, nz=256, sigma=0.5),
        # the low-fidelity side of the MFMC study, in the precision that the pipeline takes
        dict(name="lf_mixed_262144", kind="lf", precision="mixed", samples=262144, classes=10, n_y=2048),
        # the same model in its default precision, on the batch that the pilot times
        dict(name="lf_fp64_65536", kind="lf", precision="fp64", samples=65536, classes=10, n_y=2048),
        # the estimators of the study: high fidelity on 834 groups, low fidelity on 16,570, 200 replicates
        dict(name="mfmc_sobol", kind="mfmc", m1=834, m2=16570, d=3, classes=10, boot=200),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["fp64", "mixed", "mixed", "contact", "adjoint", "p3m", "lf", "mfmc"])
    if kind == "fp64":
        samples = rng.choice([1, 1, 2, 5, 16])
        n = _log(rng, 200, 40_000 // samples)
        return step_case(None, "fp64", samples, max(1, n // rng.choice([1, 3])), n, rng.choice([1, 3, 5, 10]),
                         rng.randint(2, 12), dt=rng.choice([0.05, 0.1]), sigma=rng.choice([0.0, 0.5]),
                         mode=rng.choice(["stick", "rebound"]), compact=rng.choice([0, 5, 100]))
    if kind in ("mixed", "contact"):
        contact = kind == "contact"
        n = _log(rng, 500, 16_000 if contact else 32_000)
        samples = _log(rng, 1, max(2, min(1000, int((6e9 if contact else 4e10) / n / n))))
        return step_case(None, "mixed", samples, max(1, n // rng.choice([1, 2, 8])), n, rng.choice([1, 3, 5]),
                         rng.randint(1, 10), grid=rng.choice(["small", "large"]), dt=rng.choice([0.05, 0.1]),
                         sigma=rng.choice([0.0, 0.5]), mode=rng.choice(["stick", "rebound"]), contact=contact,
                         neg=0.5 if contact else 0.0, compact=rng.choice([0, 100]))
    if kind == "adjoint":
        n = _log(rng, 200, 16_000)
        samples = _log(rng, 1, max(2, min(256, int(4e9 / n / n))))
        steps = rng.randint(3, 20)
        return dict(kind="adjoint", precision="mixed", samples=samples, count=n, classes=rng.choice([1, 3, 5]),
                    steps=steps, ckpt=rng.randint(1, steps), eps=rng.choice([0.5, 0.1]),
                    store=rng.choice([False, True]), mode=rng.choice(["stick", "rebound"]))
    if kind == "p3m":
        n = _log(rng, 20_000, 1_000_000)
        mesh, nz = (61, 128) if n <= 200_000 else (123, 256)
        return dict(kind="p3m", count=n, classes=rng.choice([5, 10]), steps=rng.randint(1, 3), mesh=mesh, nz=nz,
                    sigma=rng.choice([0.0, 0.5]))
    if kind == "lf":
        fp64 = rng.random() < 0.5
        return dict(kind="lf", precision="fp64" if fp64 else "mixed", samples=_log(rng, 64, 65_536 if fp64 else 262_144),
                    classes=rng.choice([3, 5, 10]), n_y=rng.choice([513, 1000, 2048]))
    m1 = _log(rng, 40, 2000)
    return dict(kind="mfmc", m1=m1, m2=m1 + _log(rng, 100, 40_000), d=rng.choice([2, 3]), classes=rng.choice([1, 3, 10]),
                boot=rng.choice([0, 60, 200]))


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
def _inputs(case, seed):
    """(params [S, 3], counts [S], particle and field seeds) of a case."""
    rng = np.random.Generator(np.random.Philox(seed))
    S = case.get("samples", 1)
    params = np.array([0.05, 0.5, 0.5]) * (0.5 + rng.random((S, 3)))        # +-50 % of nominal
    if "lo" in case:      # the sizes of a study are fixed; the seed draws its inputs
        counts = np.random.Generator(np.random.Philox(case["hi"])).integers(case["lo"], case["hi"] + 1, size=S)
    else:
        counts = np.full(S, case.get("count", 1))
    return params, [int(c) for c in counts], int(rng.integers(1 << 31)), int(rng.integers(1 << 31))


def _field(case, seed):
    n_r, n_th, n_z = GRIDS[case.get("grid", "large" if case["kind"] in ("p3m", "lf") else "small")]
    return pdq.Field(pdq.field_desc(n_r=n_r, n_th=n_th, n_z=n_z, n_modes=64), seed)


def _lf_params(case, seed):
    rng = np.random.Generator(np.random.Philox(seed + 1))
    return rng.random((case["samples"], 3)) * np.array([0.1, 1.0, 1.0])     # the paper's ranges


def _mfmc_tables(case, seed):
    """Pick-freeze tables of a two-model study of a smooth V_dep+-like output."""
    g = torch.Generator(device=DEV).manual_seed(seed)
    d, C, m2 = case["d"], case["classes"], case["m2"]
    x, xp = (torch.rand((m2, d), generator=g, device=DEV, dtype=torch.float64) for _ in range(2))
    cols = [x, xp]
    for j in range(d):
        z = xp.clone()
        z[:, j] = x[:, j]
        cols.append(z)
    x = torch.stack(cols, 1)                                                # [m2, d + 2, d]
    a = torch.rand((C, d), generator=g, device=DEV, dtype=torch.float64) + 0.1
    base = 1e-3 * torch.linspace(0.3, 5.0, C, device=DEV, dtype=torch.float64)
    f = base * (1.0 + (x * x) @ a.T + 0.5 * x[..., :1] * x[..., 1:2])       # [m2, d + 2, C]
    noise = torch.randn((2, m2, d + 2, C), generator=g, device=DEV, dtype=torch.float64) * 0.05 * base
    hf = (f + noise[0])[: case["m1"]].contiguous()
    lf = (0.8 * f + noise[1]).contiguous()
    return hf, lf, [case["m1"], m2], [1.0, 1.1]


def prepare(case, seed):
    kind = case["kind"]
    if kind == "mfmc":
        hf, lf, m, alpha = _mfmc_tables(case, seed)
        return dict(case=case, ys=[hf, lf], m=m, alpha=alpha, seed=seed)
    params, counts, pseed, fseed = _inputs(case, seed)
    s = dict(case=case, seed=pseed, phys=pdq.phys_default(), field=_field(case, fseed), st=st_classes(case["classes"]))
    if kind == "lf":
        s["params"] = pdq.params_tensor(_lf_params(case, seed))
        s["var"] = pdq.lf_fluid_variance(s["field"])
        s["desc"] = pdq.lf_desc(n_y=case["n_y"], precision=PRECISION[case["precision"]])
        return s
    if kind == "adjoint":
        s["params"] = torch.tensor(params, device=DEV)
        s["batch"] = pdq.Batch(PRECISION[case["precision"]], counts, s["st"])
        s["cfg"] = pdq.step_cfg(0.05, window_start=0, mode=MODES[case["mode"]])
        g = torch.Generator(device=DEV).manual_seed(seed)
        s["cotangent"] = torch.rand((len(counts), case["classes"]), generator=g, device=DEV, dtype=torch.float64) + 0.5
        return s
    s["params"] = pdq.params_tensor(params)
    s["phys"].neg_charge_frac = case.get("neg", 0.0)
    state = s["state"] = pdq.State(pdq.FP64 if kind == "p3m" else PRECISION[case["precision"]], counts, s["st"])
    s["tally"] = pdq.Tally(len(counts), len(s["st"]))
    if kind == "p3m":
        s["cfg"] = pdq.step_cfg(0.05, window_start=0, compact_every=100)
        s["plan"] = pdq.P3M(s["field"], M=case["mesh"], Nz=case["nz"], max_particles=counts[0])
    else:
        forces = pdq.F_ALL | (pdq.F_CONTACT if case["contact"] else 0)
        s["cfg"] = pdq.step_cfg(case["dt"], forces=forces, mode=MODES[case["mode"]], window_start=0,
                                compact_every=case["compact"], block=max(case["block"], 0), variant=case["variant"])
        if case["block"] < 0:
            pdq.seed_particles(s["field"], s["phys"], state, s["params"], pseed, case["sigma"])
            pdq.autotune(s["field"], s["phys"], state, s["params"], s["cfg"])
    s["ws"] = pdq.workspace(state, s["cfg"])
    # the program's own row tables, for reading the particles back by sample and id
    count = torch.tensor(counts, device=DEV)
    s["sample"] = torch.repeat_interleave(torch.arange(len(counts), device=DEV), count)
    s["first"] = state.offset[:-1][s["sample"]]
    s["row"] = torch.arange(state.st.capacity, device=DEV) - s["first"]
    return s


# ---------------------------------------------------------------------------
# One pass
# ---------------------------------------------------------------------------
def _particles(s):
    """The live particles' state in seeding order (zero rows where a particle has deposited)."""
    state = s["state"]
    n = state.st.capacity
    pos, vel, xy = state.current()
    live = (s["row"] < state.count[s["sample"]]) & (vel[:, 3] > 0.5)
    to = torch.where(live, s["first"] + state.tag[:, 0], n)
    out = {}
    for name, t in (("pos", pos), ("vel", vel), ("xy", xy)):
        if t is not None:
            out[name] = torch.zeros((n + 1, t.shape[1]), dtype=t.dtype, device=DEV)
            out[name][to] = t
            out[name] = out[name][:n]
    return out


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "mfmc":
        return pdq.mfmc_sobol(s["ys"], s["m"], s["alpha"], n_boot=case["boot"], seed=s["seed"])
    if kind == "lf":
        return {"vdep": pdq.lf_vdep(s["field"], s["phys"], s["desc"], s["var"], s["st"], s["params"])}
    if kind == "adjoint":
        params = s["params"].detach().requires_grad_(True)
        J = pdq.PdqDeposition.apply(params, s["field"], s["phys"], s["batch"], s["cfg"], case["steps"], case["ckpt"],
                                    case["eps"], s["seed"], 0.0, case["store"])
        J.backward(s["cotangent"])
        return {"J": J.detach(), "grad": params.grad}
    s["tally"].zero_()
    pdq.seed_particles(s["field"], s["phys"], s["state"], s["params"], s["seed"], case["sigma"])
    if kind == "p3m":
        pdq.step_particles_p3m(s["field"], s["phys"], s["state"], s["params"], s["cfg"], case["steps"], s["tally"],
                               s["plan"], s["ws"])
        dt = 0.05
    else:
        pdq.step_particles(s["field"], s["phys"], s["state"], s["params"], s["cfg"], case["steps"], s["tally"], s["ws"])
        dt = case["dt"]
    vdep, mean, se = pdq.deposition_tally(s["tally"], dt)
    out = _particles(s)
    out.update(n_dep=s["tally"].n_dep, n_alive=s["tally"].n_alive, vdep=vdep, mean=mean, se=se)
    return out


def _pairs(case):
    """Ordered particle pairs of one step (ragged samples: the mean of N^2 over the counts' range)."""
    if "lo" in case:
        a, b = case["lo"], case["hi"]
        return case["samples"] * (a * a + a * b + b * b) / 3.0
    return case["samples"] * float(case["count"]) ** 2


def work(case):
    kind = case["kind"]
    if kind == "mfmc":
        tables = 8.0 * (case["m1"] + case["m2"]) * (case["d"] + 2) * case["classes"]
        return {"bytes": tables, "flops": (1 + case["boot"]) * tables / 8 * 5}
    if kind == "lf":
        return {"bytes": case["samples"] * (32.0 + 8.0 * case["classes"]),
                "flops": case["samples"] * case["classes"] * (case["n_y"] - 1) * 23.0}
    if kind == "adjoint":      # forward 12 flops per ordered pair, its vector-Jacobian product 28
        n = case["samples"] * case["count"]
        return {"bytes": n * 64.0 * case["steps"] * 3, "flops": case["steps"] * (40.0 * _pairs(case) + 600.0 * n)}
    if kind == "p3m":          # transforms 5 n log2 n each of 4, short-range pairs ~40 flops each
        n, alpha_h = float(case["count"]), 0.5
        h = 2 * R_PLUS / case["mesh"]
        r_cut = 3.3 * h / alpha_h
        near = n * n * (4.0 / 3 * math.pi * r_cut ** 3) / (math.pi * R_PLUS ** 2 * L_PLUS)
        nodes = (2.0 * (case["mesh"] + 5)) ** 2 * case["nz"]
        return {"bytes": case["steps"] * (n * 136.0 + nodes * 8.0 * 4),
                "flops": case["steps"] * (40.0 * near + 4 * 5 * nodes * math.log2(nodes) + 300.0 * n)}
    n = case["samples"] * 0.5 * (case["lo"] + case["hi"])
    per = 136.0 if case["precision"] == "fp64" else 104.0
    return {"bytes": case["steps"] * n * per, "flops": case["steps"] * (12.0 * _pairs(case) + 150.0 * n)}


# ---------------------------------------------------------------------------
# The same in 64 bits, from the equations
# ---------------------------------------------------------------------------
KB = 1.380649e-23
NU, RADIUS, RE_TAU, RHO_P, RHO_F, EPS0 = 1.5e-5, 0.01, 180.0, 2650.0, 1.2, 8.854e-12
Q_UNIT, HAMAKER, DELTA_MIN, YOUNG, DELTA_C, SIGMA_Y, GRAV = (500 * 1.6e-19, 1e-18, 1e-9, 70e9, 0.165e-9, 200e6,
                                                           9.81)
USTAR = RE_TAU * NU / RADIUS
ELL, ACC, TAUF = NU / USTAR, NU / USTAR ** 3, NU / USTAR ** 2
BETA, KAPPA, B_LOG = 2.0, 0.41, 5.2


def _philox(c0, c1, c2, c3, seed):
    """Philox4x32-10 words of uint32 counter arrays under a 64-bit key."""
    c = [np.broadcast_arrays(*(np.asarray(v, np.uint64) for v in (c0, c1, c2, c3)))[k].copy() for k in range(4)]
    k0, k1 = np.uint64(seed & 0xffffffff), np.uint64((seed >> 32) & 0xffffffff)
    m0, m1, mask, sh = np.uint64(0xD2511F53), np.uint64(0xCD9E8D57), np.uint64(0xffffffff), np.uint64(32)
    for _ in range(10):
        p0, p1 = m0 * c[0], m1 * c[2]
        c = [(p1 >> sh) ^ c[1] ^ k0, p1 & mask, (p0 >> sh) ^ c[3] ^ k1, p0 & mask]
        k0, k1 = (k0 + np.uint64(0x9E3779B9)) & mask, (k1 + np.uint64(0xBB67AE85)) & mask
    return [(w.astype(np.float64) + 0.5) * 2.0 ** -32 for w in c]


def _exact_field(case, seed):
    """The gridded carrier velocity [n_z, n_th, n_r, 3]: log law plus random Fourier modes."""
    n_r, n_th, n_z = GRIDS[case.get("grid", "large" if case["kind"] in ("p3m", "lf") else "small")]
    n, lo, hi = 64, 2 * math.pi / 400.0, 2 * math.pi / 20.0
    ids = np.arange(n)
    a, b = _philox(ids, 0, 0, 1, seed), _philox(ids, 1, 0, 1, seed)
    kmag = lo * (hi / lo) ** a[0]
    ct = 2 * a[1] - 1
    st = np.sqrt(np.maximum(0, 1 - ct * ct))
    k = np.stack([kmag * st * np.cos(2 * np.pi * a[2]), kmag * st * np.sin(2 * np.pi * a[2]), kmag * ct], 1)
    dkz = 2 * np.pi / L_PLUS
    k[:, 2] = dkz * np.rint(k[:, 2] / dkz)
    kn, kp = np.linalg.norm(k, axis=1), np.hypot(k[:, 0], k[:, 1])
    e1 = np.stack([k[:, 1] / kp, -k[:, 0] / kp, np.zeros(n)], 1)
    e2 = np.cross(k / kn[:, None], e1)
    amp = math.sqrt(6.0 / n) / kn
    bv = amp[:, None] * (np.cos(2 * np.pi * a[3])[:, None] * e1 + np.sin(2 * np.pi * a[3])[:, None] * e2)
    phi = 2 * np.pi * b[0]
    f64 = dict(dtype=torch.float64, device=DEV)
    r = R_PLUS * torch.tanh(BETA * torch.arange(n_r, **f64) / (n_r - 1)) / math.tanh(BETA)
    th = 2 * math.pi * torch.arange(n_th, **f64) / n_th
    z = (L_PLUS * torch.arange(n_z, **f64) / n_z)[:, None, None]
    x, y = (torch.cos(th)[:, None] * r)[None], (torch.sin(th)[:, None] * r)[None]
    one = 1 - (x * x + y * y) / R_PLUS ** 2
    inside = (r < R_PLUS).to(torch.float64)
    f, gx, gy = one * one * inside, -4 * one * x / R_PLUS ** 2 * inside, -4 * one * y / R_PLUS ** 2 * inside
    S = [torch.zeros((n_z, n_th, n_r), **f64) for _ in range(3)]
    T = [torch.zeros((n_z, n_th, n_r), **f64) for _ in range(3)]
    kb = np.cross(k, bv)
    for m in range(n):
        arg = k[m, 0] * x + k[m, 1] * y + k[m, 2] * z + phi[m]
        ca, sa = torch.cos(arg), torch.sin(arg)
        for c in range(3):
            S[c] += ca * bv[m, c]
            T[c] += sa * kb[m, c]
    yc = 30.0
    for _ in range(100):
        yc -= (yc - math.log(yc) / KAPPA - B_LOG) / (1 - 1 / (KAPPA * yc))
    yp = torch.clamp(R_PLUS - r, min=0.0)
    mean = torch.where(yp <= yc, yp, torch.log(torch.clamp(yp, min=1e-300)) / KAPPA + B_LOG)
    return torch.stack([gy * S[2] - f * T[0], -gx * S[2] - f * T[1], gx * S[1] - gy * S[0] - f * T[2] + mean], -1)


def _classes(st):
    """Rows (tau+, d+, d, m, (d/1um)^2) of the classes."""
    rows = []
    for tau in st:
        d = math.sqrt(18.0 * RHO_F * NU * tau * TAUF / RHO_P)
        rows.append((tau, d / ELL, d, RHO_P * math.pi * d ** 3 / 6.0, (d * 1e6) ** 2))
    return torch.tensor(rows, dtype=torch.float64, device=DEV)


def _exact_seed(counts, st, seed, sigma, neg):
    """(x [n, 3], charge per unit xi, class) of the largest sample; the others are its first rows."""
    j = np.arange(max(counts))
    u = _philox(j, 0, 0, 0, seed)
    cls = torch.tensor(j % len(st), device=DEV)
    rows = _classes(st)[cls].cpu().numpy()
    lam = np.ones(len(j))
    if neg > 0:
        lam = np.where(_philox(j, 2, 0, 0, seed)[0] < neg, -1.0, 1.0)
    if sigma > 0:
        b = _philox(j, 1, 0, 0, seed)
        lam = lam * np.exp(sigma * np.sqrt(-2 * np.log(b[0])) * np.cos(2 * np.pi * b[1]))
    rr = (R_PLUS - 0.5 * rows[:, 1]) * np.sqrt(u[0])
    x = np.stack([rr * np.cos(2 * np.pi * u[1]), rr * np.sin(2 * np.pi * u[1]), L_PLUS * u[2]], 1)
    return torch.tensor(x, device=DEV), torch.tensor(rows[:, 4] * lam, device=DEV), cls


def _phi12(z):
    small = z.abs() < 0.05
    zs = torch.where(small, z, torch.zeros_like(z))
    p1, p2 = torch.zeros_like(z), torch.zeros_like(z)
    for k in range(11, -1, -1):
        p1 = p1 * zs + 1.0 / math.factorial(k + 1)
        p2 = p2 * zs + 1.0 / math.factorial(k + 2)
    zl = torch.where(small, torch.ones_like(z), z)
    em = torch.expm1(zl)
    return torch.where(small, p1, em / zl), torch.where(small, p2, (em - zl) / (zl * zl))


def _interp(grid, x):
    n_z, n_th, n_r, _ = grid.shape
    r = torch.sqrt(x[:, 0] ** 2 + x[:, 1] ** 2)
    s = torch.atanh(torch.clamp(r / R_PLUS, max=1.0) * math.tanh(BETA)) / BETA * (n_r - 1)
    i0 = torch.clamp(torch.floor(s.detach()), 0, n_r - 2).long()
    t = torch.atan2(x[:, 1], x[:, 0]) * (n_th / (2 * math.pi))
    t = torch.where(t < 0, t + n_th, t)
    j0 = torch.floor(t.detach()).long()
    zz = (x[:, 2] - L_PLUS * torch.floor(x[:, 2].detach() / L_PLUS)) * (n_z / L_PLUS)
    k0 = torch.floor(zz.detach()).long()
    tr, tt, tz = s - i0, t - j0, zz - k0
    u = 0
    for dk in (0, 1):
        for dj in (0, 1):
            for di in (0, 1):
                w = (tr if di else 1 - tr) * (tt if dj else 1 - tt) * (tz if dk else 1 - tz)
                u = u + w[:, None] * grid[(k0 + dk) % n_z, (j0 + dj) % n_th, i0 + di]
    return u


def _coulomb(x, qw, dc, rows=1 << 25):
    """sum_j qw_j d / max(|d|, dc)^3, nearest image in z, in row blocks."""
    n, out = x.shape[0], []
    step = max(1, rows // max(n, 1))
    for a in range(0, n, step):
        d = [x[a:a + step, k, None] - x[None, :, k] for k in range(3)]
        d[2] = d[2] - L_PLUS * torch.round(d[2].detach() / L_PLUS)
        r2 = torch.clamp(d[0] * d[0] + d[1] * d[1] + d[2] * d[2], min=dc * dc)
        g = qw / (r2 * torch.sqrt(r2))
        out.append(torch.stack([(g * d[k]).sum(1) for k in range(3)], 1))
    return torch.cat(out, 0)


def _contact(x, v, cls_row, alive, zeta, dt, e=0.9, steps=15.0, rows=1 << 25):
    """Collision and van der Waals accelerations between the particles of a sample, at mid-step."""
    xm = x + 0.5 * dt * v
    d_plus, d, m = cls_row[:, 1], cls_row[:, 2], cls_row[:, 3]
    near = 1.25 * float(d_plus.max())
    acc = torch.zeros_like(x)
    step = max(1, rows // len(x))
    for a in range(0, len(x), step):
        dz = xm[a:a + step, 2, None] - xm[None, :, 2]
        dz = dz - L_PLUS * torch.round(dz / L_PLUS)
        r2 = (xm[a:a + step, 0, None] - xm[None, :, 0]) ** 2 + (xm[a:a + step, 1, None] - xm[None, :, 1]) ** 2 + dz * dz
        i, j = torch.nonzero(r2 < near * near, as_tuple=True)
        dz, r2 = dz[i, j], r2[i, j]
        i = i + a
        keep = (i != j) & alive[i] & alive[j]
        i, j, dz, r = i[keep], j[keep], dz[keep], torch.sqrt(r2[keep])
        n = torch.stack([xm[i, 0] - xm[j, 0], xm[i, 1] - xm[j, 1], dz], 1) / r[:, None]
        touch = 0.5 * (d_plus[i] + d_plus[j])
        tc, le = steps * dt, math.log(e)
        vn = ((v[i] - v[j]) * n).sum(1)
        f = m[j] / (m[i] + m[j]) * ((math.pi ** 2 + le * le) / tc ** 2 * (touch - r) + 2 * le / tc * vn)
        f = torch.where(r < touch, f, torch.zeros_like(f))
        de = 2 * d[i] * d[j] / (d[i] + d[j])
        gap = (r - touch) * ELL
        g = torch.clamp(gap, min=DELTA_MIN)
        vdw = zeta * HAMAKER / 6 * de ** 6 / (g ** 2 * (2 * de + g) ** 2 * (de + g) ** 3) / m[i] * ACC
        f = f - torch.where(gap <= 0.25 * de, vdw, torch.zeros_like(vdw))
        acc.index_add_(0, i, f[:, None] * n)
    return acc


def _advance(grid, rows, x, v, q, qw, dc, prm, dt, extra=None, act=None):
    """Positions and velocities after one step, before the wall contact."""
    coef = (Q_UNIT ** 2 / (4 * math.pi * EPS0) / rows[:, 3] / ELL ** 2 * ACC)[:, None]
    a = coef * q[:, None] * _coulomb(x, qw, dc)
    a = a + torch.tensor([0.0, 0.0, GRAV * ACC], dtype=torch.float64, device=DEV)
    if extra is not None:
        a = a + extra
    r = torch.sqrt(x[:, 0] ** 2 + x[:, 1] ** 2)
    yw = torch.maximum(R_PLUS - r, 0.5 * rows[:, 1])
    aw = 0.25 * coef[:, 0] * q * q / (yw * yw)
    gap = (R_PLUS - r - 0.5 * rows[:, 1]) * ELL
    d, dl = rows[:, 2], torch.clamp(gap, min=DELTA_MIN)
    vdw = prm[1] * HAMAKER / (3 * rows[:, 3]) * ACC * d ** 6 / (dl ** 2 * (2 * d + dl) ** 2 * (d + dl) ** 3)
    aw = (aw + torch.where(gap <= 0.25 * d, vdw, torch.zeros_like(vdw)))[:, None]
    a = a + torch.cat([aw * x[:, :2] / r[:, None], torch.zeros_like(aw)], 1)
    u = _interp(grid, x)
    w = u - v
    re = torch.sqrt((w * w).sum(1)) * rows[:, 1]
    lam = ((1 + 0.15 * re ** 0.687) / rows[:, 0])[:, None]
    z = -lam * dt
    p1, p2 = _phi12(z)
    F = lam * u + a
    xn = x + v * dt * p1 + F * dt * dt * p2
    vn = v * torch.exp(z) + F * dt * p1
    return torch.cat([xn[:, :2], (xn[:, 2] - L_PLUS * torch.floor(xn[:, 2].detach() / L_PLUS))[:, None]], 1), vn


def _rebound(rows, x, v, prm, smooth):
    """(x, v, energy argument) with the particles at the wall reflected by the restitution model."""
    gc = prm[1] * HAMAKER / (24 * math.pi * DELTA_C ** 2)
    arg = (SIGMA_Y * (1 - prm[2])) ** 2 / (RHO_P * YOUNG) - 2 * (math.pi * rows[:, 2] ** 2 / 4) * gc / rows[:, 3]
    r = torch.sqrt(x[:, 0] ** 2 + x[:, 1] ** 2)
    hit = R_PLUS - r - 0.5 * rows[:, 1] <= 0
    if not smooth:
        hit = hit & (arg > 0)
    n = x[:, :2] / r[:, None]
    vn = (v[:, :2] * n).sum(1)
    cor = torch.sqrt(torch.clamp(arg, min=1e-300)) / torch.where(vn > 0, vn * USTAR, torch.ones_like(vn))
    cor = torch.where(vn > 0, torch.clamp(cor, max=1.0), torch.ones_like(vn))
    cor = torch.where(arg > 0, cor, torch.zeros_like(cor))
    dv = (-cor * vn.abs() - vn)[:, None] * n
    xr = n * (2 * (R_PLUS - 0.5 * rows[:, 1]) - r)[:, None]
    h = hit[:, None]
    x = torch.cat([torch.where(h, xr, x[:, :2]), x[:, 2:]], 1)
    v = torch.cat([torch.where(h, v[:, :2] + dv, v[:, :2]), v[:, 2:]], 1)
    return x, v, arg


def _exact_step(case, seed):
    if case["steps"] * _pairs(case) > 2.5e10:
        return None
    params, counts, pseed, fseed = _inputs(case, seed)
    st = st_classes(case["classes"])
    grid, rows = _exact_field(case, fseed), _classes(st)
    x0, qhat, cls0 = _exact_seed(counts, st, pseed, case["sigma"], case["neg"])
    dc = float(rows[:, 1].max())
    out = {"pos": [], "vel": [], "xy": []}
    n_dep, n_alive = (np.zeros((len(counts), len(st)), np.int64) for _ in range(2))
    for s, n in enumerate(counts):
        x, q, cls = x0[:n].clone(), params[s, 0] * qhat[:n], cls0[:n]
        v, alive, cr = torch.zeros_like(x), torch.ones(n, dtype=torch.bool, device=DEV), rows[cls0[:n]]
        for _ in range(case["steps"]):
            extra = _contact(x, v, cr, alive, params[s, 1], case["dt"]) if case["contact"] else None
            xn, vn = _advance(grid, cr, x, v, q, q * alive, dc, params[s], case["dt"], extra)
            r = torch.sqrt(xn[:, 0] ** 2 + xn[:, 1] ** 2)
            dep = alive & (R_PLUS - r - 0.5 * cr[:, 1] <= 0)
            if case["mode"] == "rebound":
                xn, vn, arg = _rebound(cr, xn, vn, params[s], False)
                dep = dep & ~(arg > 0)
            n_alive[s] += torch.bincount(cls[alive], minlength=len(st)).cpu().numpy()
            n_dep[s] += torch.bincount(cls[dep], minlength=len(st)).cpu().numpy()
            x, v = torch.where(alive[:, None], xn, x), torch.where(alive[:, None], vn, v)
            alive = alive & ~dep
        live = alive[:, None].to(torch.float64)
        out["pos"].append(torch.cat([x, q[:, None]], 1) * live)
        out["vel"].append(torch.cat([v, torch.ones_like(live)], 1) * live)
        out["xy"].append(x[:, :2] * live)
    out = {k: torch.cat(t, 0) for k, t in out.items() if not (k == "xy" and case["precision"] == "fp64")}
    vdep = np.where(n_alive > 0, 0.5 * R_PLUS / case["dt"] * n_dep / np.maximum(n_alive, 1), 0.0)
    se = vdep.std(0, ddof=1) / math.sqrt(len(vdep)) if len(vdep) > 1 else np.zeros(len(st))
    out.update(n_dep=n_dep, n_alive=n_alive, vdep=vdep, mean=vdep.mean(0), se=se)
    return out


def _exact_adjoint(case, seed):
    if case["steps"] * _pairs(case) > 4e9:
        return None
    params, counts, pseed, fseed = _inputs(case, seed)
    st = st_classes(case["classes"])
    C, dt = len(st), 0.05
    grid, rows = _exact_field(case, fseed), _classes(st)
    x0, qhat, cls0 = _exact_seed(counts, st, pseed, 0.0, 0.0)
    dc = float(rows[:, 1].max())
    g = torch.Generator(device=DEV).manual_seed(seed)
    cot = torch.rand((len(counts), C), generator=g, device=DEV, dtype=torch.float64) + 0.5
    Js, grads = [], []
    for s, n in enumerate(counts):
        prm = torch.tensor(params[s], device=DEV, requires_grad=True)
        cls, cr = cls0[:n], rows[cls0[:n]]
        hot = torch.nn.functional.one_hot(cls, C).to(torch.float64)

        def step(x, v, w, prm):
            q = prm[0] * qhat[:n]
            x, v = _advance(grid, cr, x, v, q, q * w, dc, prm, dt)
            gap = R_PLUS - torch.sqrt(x[:, 0] ** 2 + x[:, 1] ** 2) - 0.5 * cr[:, 1]
            p = torch.sigmoid(-gap / case["eps"])
            if case["mode"] == "rebound":
                x, v, arg = _rebound(cr, x, v, prm, True)
                p = p * torch.sigmoid(-arg / 10.0)
            return x, v, w * (1 - p)

        x, v, w = x0[:n].clone(), torch.zeros((n, 3), dtype=torch.float64, device=DEV), torch.ones(n, dtype=torch.float64,
                                                                                                     device=DEV)
        num, den = 0, 0
        for _ in range(case["steps"]):
            x, v, wn = torch.utils.checkpoint.checkpoint(step, x, v, w, prm, use_reentrant=False)
            num, den, w = num + (w - wn) @ hot, den + w @ hot, wn
        J = 0.5 * R_PLUS * num / (dt * den)
        (gr,) = torch.autograd.grad((J * cot[s]).sum(), prm, allow_unused=True)
        Js.append(J.detach())
        grads.append(gr)
    return {"J": torch.stack(Js), "grad": torch.stack(grads)}


def _exact_lf(case, seed):
    _, _, _, fseed = _inputs(case, seed)
    grid = _exact_field(case, fseed)
    th = 2 * math.pi * torch.arange(grid.shape[1], dtype=torch.float64, device=DEV) / grid.shape[1]
    ur = torch.cos(th)[None, :, None] * grid[..., 0] + torch.sin(th)[None, :, None] * grid[..., 1]
    var = ur.var(dim=(0, 1), unbiased=False).cpu().numpy()
    prm = torch.tensor(_lf_params(case, seed), device=DEV)
    rows = _classes(st_classes(case["classes"])).cpu().numpy()
    TL, temp, cut, n = 10.0, 293.15, 1e-12 / ELL, case["n_y"]
    cell = np.zeros((n - 1, 5, len(rows)))
    sg, K0 = np.zeros(len(rows)), []
    for c, (tau, dp, d, m, qf) in enumerate(rows):
        s = np.arange(n) / (n - 1)
        yw = 0.5 * dp
        y = yw + (R_PLUS - yw) * np.expm1(8.0 * s) / np.expm1(8.0)
        t = np.arctanh((R_PLUS - y) * math.tanh(BETA) / R_PLUS) / BETA * (len(var) - 1)
        i = np.clip(np.floor(t).astype(int), 0, len(var) - 2)
        vf = (1 - (t - i)) * var[i] + (t - i) * var[i + 1]
        w, D = TL / (TL + tau) * vf, KB * temp * tau * TAUF / m / NU + vf * TL
        gap = y - yw
        psi = np.where(gap >= cut, 1 / np.maximum(gap, cut), 2 / cut - gap / cut ** 2)
        ce = 3 * (Q_UNIT * qf) ** 2 / (8 * math.pi ** 2 * EPS0 * RHO_P * d ** 3) * ACC / ELL ** 2
        cv = HAMAKER * d / (12 * m) * ACC / ELL ** 2
        dy = np.diff(y)
        cell[:, :, c] = np.stack([np.diff(w), -ce * np.diff(1 / y), -cv * np.diff(psi), dy / tau,
                                  dy / (0.5 * (D[1:] + D[:-1]))], 1)
        sg[c] = math.sqrt(w[0] + KB * temp / m / USTAR ** 2)
    cell, sg = torch.tensor(cell, device=DEV), torch.tensor(sg, device=DEV)
    xi2, zeta = prm[:, :1] ** 2, prm[:, 1:2]
    V = torch.zeros((len(prm), len(rows)), dtype=torch.float64, device=DEV)
    P, Q = torch.ones_like(V), torch.zeros_like(V)
    for k in range(n - 2, -1, -1):
        dw, de, dv, a, h = cell[k]
        c = 0.5 * V * V + dw + (xi2 * de + zeta * dv)
        root = -2 * c / (a + torch.sqrt(a * a + 2 * torch.clamp(c, min=0.0)))
        Vi = torch.where(c > 0, root, torch.zeros_like(root))
        am = 0.5 * (V + Vi) * h
        em = torch.expm1(am)
        G = torch.where(am != 0, h * em / torch.where(am != 0, am, torch.ones_like(am)), h.expand_as(am))
        Q = Q + P * G
        P = P * (1 + em)
        V = Vi
    u = -V
    M = u / (math.sqrt(2.0) * sg)
    K = -(0.5 * u * (1 + torch.erf(M)) + sg * torch.exp(-M * M) / math.sqrt(2 * math.pi))
    return {"vdep": -K / (P - K * Q)}


def _exact_mfmc(case, seed):
    hf, lf, m, alpha = _mfmc_tables(case, seed)
    d, C = case["d"], case["classes"]
    mean, var, V, T = np.zeros(C), np.zeros(C), np.zeros((d, C)), np.zeros((d, C))
    for y, n, w in ((hf, m[0], 1.0), (lf, m[1], alpha[1]), (lf, m[0], -alpha[1])):
        y = y[:n].cpu().numpy()
        E, Ep, v, vp = y[:, 0].mean(0), y[:, 1].mean(0), y[:, 0].var(0, ddof=1), y[:, 1].var(0, ddof=1)
        mean += w * E
        var += w * v
        for j in range(d):
            V[j] += w * 2 * n / (2 * n - 1) * ((y[:, 0] * y[:, 2 + j]).mean(0) - 0.25 * (E + Ep) ** 2 + (v + vp) / (4 * n))
            T[j] += w * ((y[:, 1] - y[:, 2 + j]) ** 2).sum(0) / (2 * n)
    out = {"mean": mean, "var": var, "s_main": V / var, "s_total": T / var}
    if case["boot"]:
        out.update(s_main_ci=None, s_total_ci=None)
    return out


def exact(case, seed):
    if case["kind"] == "p3m":      # an approximation of sums over a million particles and their images
        return None
    return {"step": _exact_step, "adjoint": _exact_adjoint, "lf": _exact_lf, "mfmc": _exact_mfmc}[case["kind"]](case, seed)
