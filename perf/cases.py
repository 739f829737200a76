"""Measured cases of the library: what a user of pmf.h / pmf.py has it do.

Every case goes through the Python binding (the C ABI's own names).  The
sizes are those of the repository's workloads (the 104-bead chain with 21
windows, the uneven batch of 40-400 beads, the 1D double well, the reductions
of their sample stores, the surrogate's training) and a range around them,
from which draw() takes more.

A chain pass is a few hundred steps long: FP32 trajectories that differ by
rounding separate by about a factor e per 100 steps, so longer ones have no
common result to compare.  What a pass returns is what the protocol goes on
with: the x samples (the estimators' input) and, where a run is continued,
the end positions (the start of a seeded run, whose velocities are drawn
anew).  FP32 runs hand their end positions out as doubles holding FP32
values; they are given back here as the FP32 numbers they are.
"""
import math

import numpy as np
import torch

from paper_1105_4840_gb300 import inputs, pmf

KT300 = inputs.kT_of(300.0)
FIELDS = pmf.RESULT_FIELDS


# --------------------------------------------------------------------------
# the cases
# --------------------------------------------------------------------------

def listed():
    return [
        # the parallel protocol on the 104-bead chain at the benchmark's counts
        dict(name="chain104_ppp", kind="chain", beads=104, windows=21, replicas=32, steps=400, stride=10, warps=0,
             fp64=False, final=False),
        # a first look at a path: few replicas, the GPU mostly empty; end
        # positions are read back to continue the windows
        dict(name="chain104_few", kind="chain", beads=104, windows=21, replicas=8, steps=240, stride=20, warps=0,
             fp64=False, final=True),
        # a short peptide-sized chain with more replicas per window
        dict(name="chain40_wide", kind="chain", beads=40, windows=21, replicas=64, steps=300, stride=10, warps=0,
             fp64=False, final=False),
        # the 200-bead chain of the placement study at the warp count its
        # launches use when replicas are scarce; odd length, ragged tile
        dict(name="chain201_long", kind="chain", beads=201, windows=21, replicas=16, steps=200, stride=25, warps=8,
             fp64=False, final=True),
        # many uneven chains in one packed launch
        dict(name="batch_uneven", kind="batch", chains=12, n_min=40, n_max=400, w_min=21, w_max=61, replicas=16,
             steps=200, stride=20),
        # FP64 integration, the reference arm of the precision study
        dict(name="chain104_fp64", kind="chain", beads=104, windows=21, replicas=8, steps=100, stride=10, warps=0,
             fp64=True, final=True),
        # the whole 1D workload: simulation and estimates
        dict(name="od1d_ppp", kind="od1d", windows=21, replicas=8, steps=20000, stride=10),
        # constant-velocity pulling of the 1D model with its estimates
        dict(name="od1d_pull", kind="pull1d", replicas=256, steps=4400, stride=10),
        # one step's estimates of the 104-bead workload's sample store
        dict(name="reduce_ppp", kind="reduce", windows=21, replicas=32, samples=3600),
        # the smallest call: estimates of a short path in a monitoring loop
        dict(name="reduce_small", kind="reduce", windows=5, replicas=4, samples=256),
        # a large store, bound by memory: odd sample count
        dict(name="reduce_large", kind="reduce", windows=64, replicas=512, samples=1801),
        # the surrogate's training in one round of the window placement
        dict(name="surrogate_train", kind="surrogate", windows=21, replicas=8, steps=200, batch=512),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["chain", "chain", "chain", "chain", "batch", "fp64", "od1d", "pull1d", "reduce", "reduce", "reduce",
                       "surrogate"])
    if kind in ("chain", "fp64"):
        fp64 = kind == "fp64"
        n = _log_int(rng, 40, 150 if fp64 else 400)
        w = rng.randint(5, 61)
        r = _log_int(rng, 2, 16 if fp64 else 64)
        steps = rng.randrange(40, 101, 10) if fp64 else rng.randrange(100, 241, 20)
        room = (2e9 if fp64 else 3e10) / (n * n * w * steps)
        return dict(kind="chain", beads=n, windows=w, replicas=max(1, min(r, int(room))), steps=steps,
                    stride=rng.choice([5, 7, 10, 20]), warps=0 if fp64 else rng.choice([0, 0, 4, 5, 6, 8]), fp64=fp64,
                    final=rng.random() < 0.5)
    if kind == "batch":
        return dict(kind="batch", chains=rng.randint(3, 10), n_min=40, n_max=rng.randint(100, 400), w_min=5,
                    w_max=rng.randint(15, 50), replicas=_log_int(rng, 2, 16), steps=rng.randrange(100, 201, 20), stride=20)
    if kind == "od1d":
        return dict(kind="od1d", windows=rng.randint(5, 41), replicas=_log_int(rng, 2, 128),
                    steps=_log_int(rng, 500, 20000), stride=rng.choice([1, 7, 10, 25]))
    if kind == "pull1d":
        return dict(kind="pull1d", replicas=_log_int(rng, 16, 2048), steps=_log_int(rng, 550, 20000),
                    stride=rng.choice([7, 10, 25]))
    if kind == "reduce":
        w, t = rng.randint(2, 100), _log_int(rng, 60, 4000)
        r = min(_log_int(rng, 2, 600), 65536 // w, max(2, 60_000_000 // (w * t)))
        return dict(kind="reduce", windows=w, replicas=r, samples=t)
    return dict(kind="surrogate", windows=rng.randint(7, 41), replicas=_log_int(rng, 2, 32),
                steps=rng.randint(40, 200), batch=128 * rng.randint(1, 8))


# --------------------------------------------------------------------------
# inputs
# --------------------------------------------------------------------------

def _f32(a):
    return np.asarray(a, dtype=np.float64).astype(np.float32).astype(np.float64)


def _settings(case, seed, k, kT, dt, gamma):
    equil = case["steps"] // 10
    return inputs.RunSettings(k=k, kT=kT, dt=dt, gamma=gamma, n_steps=case["steps"], n_equil=equil,
                              stride=case["stride"], replicas=case["replicas"], seed=seed & 0x7FFFFFFF)


def _chain_path(n, windows):
    scale = math.sqrt(n / 104.0)  # a random coil's size grows about as sqrt(N)
    return inputs.lambda_grid(1.3 * scale, 3.3 * scale, windows)


def _chain_inputs(case, seed):
    p = inputs.chain_params(case["beads"], seed)
    lam = _chain_path(case["beads"], case["windows"])
    start = _f32(inputs.chain_start(p, seed + 1000, target_x=lam[0], tries=4))
    return p, start, lam, _settings(case, seed, 500.0, KT300, 0.001, 5.0)


def _batch_inputs(case, seed):
    g = np.random.Generator(np.random.PCG64(seed))
    # the lengths and window counts are the case's, not the seed's: evenly
    # spread over their ranges, odd and even ones mixed
    c = case["chains"]
    lengths = [int(round(case["n_min"] + (case["n_max"] - case["n_min"]) * i / (c - 1))) for i in range(c)]
    windows = [int(round(case["w_min"] + (case["w_max"] - case["w_min"]) * ((5 * i) % c) / (c - 1))) for i in range(c)]
    params = [inputs.chain_params(n, int(g.integers(1 << 30))) for n in lengths]
    starts = [_f32(inputs.chain_start(p, int(g.integers(1 << 30)), tries=8)) for p in params]
    lams = [_chain_path(n, w) for n, w in zip(lengths, windows)]
    return params, starts, lams, _settings(case, seed, 500.0, KT300, 0.001, 5.0)


def _well(case, seed):
    run = _settings(case, seed, 20.0, 1.0, 1e-3, 1.0)
    return run, inputs.lambda_grid(-1.5, 1.5, case.get("windows", 21))


def _store(case, seed):
    """Samples [windows][replicas][samples] around the windows' centres, lagging
    behind them as a pulled chain does."""
    w, r, t = case["windows"], case["replicas"], case["samples"]
    g = torch.Generator(device="cuda").manual_seed(seed)
    lam = torch.from_numpy(inputs.lambda_grid(1.3, 3.3, w)).cuda()
    x = torch.randn((w, r, t), generator=g, device="cuda", dtype=torch.float32)
    x *= math.sqrt(1.2 * KT300 / 500.0)
    x += (lam - 0.1 * (torch.arange(w, device="cuda") % 3)).float()[:, None, None]
    return x, lam


PULL = dict(lambda1=-1.2, velocity=0.5)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "chain":
        p, start, lam, run = _chain_inputs(case, seed)
        system = pmf.pmf_create_system_chain([p], [start], precision=pmf.PMF_FP64 if case["fp64"] else pmf.PMF_FP32)
        if case["warps"]:
            pmf.pmf_chain_set_warps(system, 0, case["warps"])
        return dict(case=case, run=pmf.pmf_run_prepare(system, lam, pmf.make_params(run)))
    if kind == "batch":
        params, starts, lams, run = _batch_inputs(case, seed)
        system = pmf.pmf_create_system_chain(params, starts)
        return dict(case=case, run=pmf.pmf_run_batch_prepare(system, list(enumerate(lams)), pmf.make_params(run)))
    if kind in ("od1d", "pull1d"):
        run, lam = _well(case, seed)
        system = pmf.pmf_create_system_1d(2.0, -1.0)
        prm = pmf.make_params(run)
        rr = (pmf.pmf_run_prepare(system, lam, prm) if kind == "od1d"
              else pmf.pmf_run_prepare_smd(system, PULL["lambda1"], PULL["velocity"], prm))
        return dict(case=case, run=rr)
    if kind == "reduce":
        x, lam = _store(case, seed)
        out = torch.zeros((len(FIELDS), case["windows"]), dtype=torch.float64, device="cuda")
        # the caller reads the fields where the call leaves them
        return dict(case=case, x=x, lam=lam, out=out, fields={f: out[i] for i, f in enumerate(FIELDS)})
    # the store the surrogate learns from: a finished 1D run
    run, lam = _well(dict(case, steps=20000, stride=10), seed)
    rr = pmf.pmf_run_windows(pmf.pmf_create_system_1d(2.0, -1.0), lam, pmf.make_params(run))
    w0 = pmf.pack_mlp_params(inputs.mlp_init_params(seed & 0xFFFF))
    return dict(case=case, run=rr, mlp=pmf.Mlp(w0, 0.0, 1.5), seed=seed & 0x7FFFFFFF)


def _flat(xs):
    """The sample store behind x_samples()'s per-window views."""
    return xs[0].base


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "reduce":
        pmf.pmf_free_energy_noalloc(state["x"].data_ptr(), state["lam"].data_ptr(), case["windows"], case["replicas"],
                                    case["samples"], 500.0, KT300, state["out"].data_ptr())
        return state["fields"]
    if kind == "surrogate":
        loss = state["mlp"].train(state["run"], case["steps"], case["batch"], 3e-3, state["seed"])
        return {"params": state["mlp"].params(), "loss": loss}
    rr = state["run"]
    rr.launch()
    rr.wait()
    out = {"x": _flat(rr.x_samples())}
    if kind == "chain" and case["final"]:
        pos = rr.final_state()[0]
        out["pos"] = pos if case["fp64"] else pos.astype(np.float32)
    elif kind == "od1d":
        out["pos"] = rr.final_state()[0]
        out["fe"] = rr.free_energy()
    elif kind == "pull1d":
        out["work"] = rr.smd_work()
        out["fe"] = rr.smd_free_energy()
    return out


# --------------------------------------------------------------------------
# what a pass cannot do without
# --------------------------------------------------------------------------

def _chain_flops(n):
    """One BAOAB step of an n-bead chain (FMA = 2): 36 per nonbonded pair
    (|i - j| >= 3), 20 per bond, 60 per angle, 110 per dihedral, 33 per bead."""
    pairs = n * (n - 1) // 2 - (2 * n - 3)
    return 36 * pairs + 20 * (n - 1) + 60 * (n - 2) + 110 * (n - 3) + 33 * n


def _records(case):
    return (case["steps"] - case["steps"] // 10) // case["stride"]


def work(case):
    kind = case["kind"]
    if kind == "chain":
        sims, n = case["windows"] * case["replicas"], case["beads"]
        real = 8 if case["fp64"] else 4
        return {"bytes": 4 * sims * _records(case) + (sims * n * 3 * real if case["final"] else 0) + n * 13 * real,
                "flops": sims * case["steps"] * _chain_flops(n)}
    if kind == "batch":
        c = case["chains"]
        b = f = 0
        for i in range(c):
            n = int(round(case["n_min"] + (case["n_max"] - case["n_min"]) * i / (c - 1)))
            w = int(round(case["w_min"] + (case["w_max"] - case["w_min"]) * ((5 * i) % c) / (c - 1)))
            b += 4 * w * case["replicas"] * _records(case) + 52 * n
            f += w * case["replicas"] * case["steps"] * _chain_flops(n)
        return {"bytes": b, "flops": f}
    if kind in ("od1d", "pull1d"):
        # 8 flops a step (five of the update, three of the trap and noise term)
        sims = case["replicas"] * case.get("windows", 1)
        return {"bytes": (12 if kind == "pull1d" else 4) * sims * _records(case) + 8 * sims,
                "flops": 8 * sims * case["steps"]}
    if kind == "reduce":
        n = case["windows"] * case["replicas"] * case["samples"]
        # an exponential (20) and two sums of moments per sample
        return {"bytes": 4 * n + 8 * 15 * case["windows"], "flops": 26 * n}
    # three 64 x 64 products per sample and the Adam update of every weight
    return {"bytes": 4 * 2 * pmf.PMF_MLP_PARAMS + 4 * case["steps"] * case["batch"],
            "flops": case["steps"] * (case["batch"] * 3 * 2 * 64 * 64 + 12 * pmf.PMF_MLP_PARAMS)}


# --------------------------------------------------------------------------
# the same in 64 bits, with torch alone
# --------------------------------------------------------------------------

def _philox(c0, c1, c2, c3, seed):
    """Philox4x32-10 words (int64 tensors holding 32-bit values)."""
    m = 0xFFFFFFFF
    k0, k1 = seed & m, (seed >> 32) & m

    def mul(a, x):
        # 32 x 32 -> 64 bits by halves of x (a 64-bit product would overflow)
        lo, hi = a * (x & 0xFFFF), a * (x >> 16)
        t = (lo >> 16) + hi
        return t >> 16, ((t & 0xFFFF) << 16) | (lo & 0xFFFF)

    for _ in range(10):
        h0, l0 = mul(0xD2511F53, c0)
        h1, l1 = mul(0xCD9E8D57, c2)
        c0, c1, c2, c3 = h1 ^ c1 ^ k0, l1, h0 ^ c3 ^ k1, l0
        k0, k1 = (k0 + 0x9E3779B9) & m, (k1 + 0xBB67AE85) & m
    return c0, c1, c2, c3


def _normals(block, uid, step, tag, seed):
    """Box-Muller normals [..., 4] of the Philox blocks (block, uid, step, tag)."""
    block, uid, step = torch.broadcast_tensors(block, uid, step)
    w = _philox(block, uid, step, torch.full_like(block, tag), seed)
    u = [(v.double() + 0.5) * 2.0 ** -32 for v in w]
    r0, r1 = torch.sqrt(-2.0 * torch.log(u[0])), torch.sqrt(-2.0 * torch.log(u[2]))
    a0, a1 = 2.0 * math.pi * u[1], 2.0 * math.pi * u[3]
    return torch.stack([r0 * torch.cos(a0), r0 * torch.sin(a0), r1 * torch.cos(a1), r1 * torch.sin(a1)], -1)


class _Forces:
    """-grad H of B replicas of one chain, positions [B, 3, N]."""

    def __init__(self, p, k):
        d = lambda a: torch.from_numpy(np.ascontiguousarray(a, dtype=np.float64)).cuda()  # noqa: E731
        n, s, e, q = p.n, d(p.sigma), d(p.epsilon), d(p.charge)
        i = torch.arange(n, device="cuda")
        on = ((i[:, None] - i[None, :]).abs() >= 3).double() * float(p.nonbonded)
        self.s2 = (0.5 * (s[:, None] + s[None, :])) ** 2
        self.e24 = 24.0 * torch.sqrt(e[:, None] * e[None, :]) * on
        self.qq = p.ke * q[:, None] * q[None, :] * on
        self.eye = torch.eye(n, device="cuda", dtype=torch.float64)
        self.p, self.k = p, k
        self.kc = d(p.dih_k * np.cos(p.dih_phase))[: n - 3]

    def __call__(self, x, lam):
        dx = x[:, :, None, :] - x[:, :, :, None]  # [B, 3, i, j] = x_j - x_i
        r2 = dx.square().sum(1).add_(self.eye)
        inv2 = 1.0 / r2
        y = (self.s2 * inv2) ** 3
        fr = (self.qq * torch.rsqrt(r2) + self.e24 * y * (2.0 * y - 1.0)).mul_(inv2)
        f = -torch.einsum("bij,bcij->bci", fr, dx)
        return f + self.bonded(x, lam)

    def bonded(self, x, lam):
        p = self.p
        with torch.enable_grad():
            x = x.detach().requires_grad_(True)
            b = x[:, :, 1:] - x[:, :, :-1]
            l2 = b.square().sum(1)
            u = 0.5 * p.kb * (torch.sqrt(l2) - p.r0).square().sum()
            cs = -(b[:, :, :-1] * b[:, :, 1:]).sum(1) / torch.sqrt(l2[:, :-1] * l2[:, 1:])
            u = u + 0.5 * p.ktheta * (torch.acos(cs.clamp(-1.0, 1.0)) - p.theta0).square().sum()
            nrm = torch.cross(b[:, :, :-1], b[:, :, 1:], dim=1)
            n2 = nrm.square().sum(1)
            c = (nrm[:, :, :-1] * nrm[:, :, 1:]).sum(1) / torch.sqrt(n2[:, :-1] * n2[:, 1:])
            u = u + (self.kc[:, 0] * c + self.kc[:, 1] * (2 * c * c - 1) + self.kc[:, 2] * (4 * c ** 3 - 3 * c)).sum()
            xe = torch.sqrt((x[:, :, -1] - x[:, :, 0]).square().sum(1))
            u = u + 0.5 * self.k * (xe - lam).square().sum()
            return -torch.autograd.grad(u, x)[0]


def _chain_exact(p, start, lam, run, uid0, final):
    """BAOAB from `start` in every window and replica: samples and end positions."""
    n, R = p.n, run.replicas
    B = lam.size * R
    force = _Forces(p, run.k)
    lam_b = torch.from_numpy(np.repeat(lam, R)).cuda()
    im = torch.from_numpy(1.0 / p.mass).cuda()
    sv = torch.sqrt(run.kT * im)
    c1 = math.exp(-run.gamma * run.dt)
    c2 = math.sqrt(1.0 - c1 * c1)
    blocks = torch.arange((3 * n + 3) // 4, device="cuda")
    uid = uid0 + torch.arange(B, device="cuda")

    def noise(step, tag):  # [B, 3, n]
        z = _normals(blocks, uid[:, None], torch.tensor(step, device="cuda"), tag, run.seed)
        return z.reshape(B, -1)[:, : 3 * n].reshape(B, n, 3).transpose(1, 2)

    x = torch.from_numpy(start).cuda().T[None].repeat(B, 1, 1)
    v = sv * noise(0, 1)
    h = 0.5 * run.dt
    out = []
    f = force(x, lam_b)
    for step in range(run.n_steps):
        v = v + h * f * im
        x = x + h * v
        v = c1 * v + c2 * sv * noise(step, 0)
        x = x + h * v
        f = force(x, lam_b)
        v = v + h * f * im
        done = step + 1 - run.n_equil
        if done > 0 and done % run.stride == 0:
            out.append(torch.sqrt((x[:, :, -1] - x[:, :, 0]).square().sum(1)))
    xs = torch.stack(out, 1).cpu().numpy()  # [B, T]
    return xs, x.transpose(1, 2).reshape(-1).cpu().numpy() if final else None


def _profile(x, lam, k, kT):
    """The estimators over x [windows, replicas, samples] (64-bit tensor)."""
    s, R, T = x.shape
    d = torch.zeros_like(lam)
    d[:-1] = lam[1:] - lam[:-1]
    e = x - lam[:, None, None]
    a = e.sum(2)
    n = float(R * T)
    mean_e = a.sum(1) / n
    var = (e - mean_e[:, None, None]).square().mean((1, 2))
    del e
    w = 0.5 * k * d[:, None, None] * ((2 * lam + d)[:, None, None] - 2.0 * x)
    m = w.amin((1, 2))
    E = torch.exp(-(w - m[:, None, None]) / kT).sum(2)
    del w
    je = m - kT * torch.log(E.sum(1) / n)
    fl = -k * d * mean_e
    g2 = k * var / kT
    loo = m[:, None] - kT * torch.log((E.sum(1, keepdim=True) - E) / (n - T))
    lof = -(k * d)[:, None] * (a.sum(1, keepdim=True) - a) / (n - T)
    jk = lambda q: (R - 1.0) / R * (q - q.mean(1, keepdim=True)).square().sum(1)  # noqa: E731

    def upto(q):
        return torch.cat([torch.zeros(1, device=q.device, dtype=q.dtype), torch.cumsum(q[:-1], 0)])

    r = {"lambda": lam, "dF_JE": upto(je), "dF_fluct": upto(fl),
         "dF_G": upto(0.5 * k * d * d * (1.0 - g2) + fl), "W_mean": upto(0.5 * k * d * (d - 2.0 * mean_e)),
         "se_JE": torch.sqrt(upto(jk(loo))), "se_fluct": torch.sqrt(upto(jk(lof))),
         "mean_x": lam + mean_e, "var_x": var, "gamma2": g2}
    vw = upto((k * d).square() * var)
    r["var_ZW"] = vw / n + vw * vw / (2.0 * kT * kT * (n - 1.0))
    r["var_ZW"][0] = 0.0
    r["dF_com"], r["uncertainty"] = 0.5 * (r["dF_JE"] + r["dF_fluct"]), 0.5 * (r["dF_JE"] - r["dF_fluct"])
    span = lam - lam[0]
    span[0] = 1.0
    r["acc_force"] = r["dF_fluct"] / span
    return {f: r[f].cpu().numpy() for f in FIELDS}


def _well_exact(case, seed):
    run, lam = _well(case, seed)
    pull = case["kind"] == "pull1d"
    R = run.replicas
    B = R if pull else lam.size * R
    uid = torch.arange(B, device="cuda")
    lam_b = torch.full((B,), PULL["lambda1"], device="cuda", dtype=torch.float64) if pull else \
        torch.from_numpy(np.repeat(lam, R)).cuda()
    x = torch.full((B,), -1.0, device="cuda", dtype=torch.float64)
    W = torch.zeros_like(x)
    amp = math.sqrt(2.0 * run.kT * run.dt / run.gamma)
    xs, ws = [], []
    for n0 in range(0, run.n_steps, 1024):
        blocks = torch.arange(n0 // 4, n0 // 4 + 256, device="cuda")
        z = amp * _normals(torch.zeros_like(blocks), uid[:, None], blocks, 0, run.seed).reshape(B, -1).T.contiguous()
        for j in range(min(1024, run.n_steps - n0)):
            step = n0 + j
            if pull and step > run.n_equil:
                old, lam_b = lam_b, PULL["lambda1"] + PULL["velocity"] * run.dt * (step - run.n_equil) + 0.0 * x
                W = W + 0.5 * run.k * (lam_b - old) * (lam_b + old - 2.0 * x)
            x = x + (-8.0 * x * (x * x - 1.0) - run.k * (x - lam_b)) * (run.dt / run.gamma) + z[j]
            done = step + 1 - run.n_equil
            if done > 0 and done % run.stride == 0:
                xs.append(x)
                ws.append(W)
    X, Wr = torch.stack(xs, 1), torch.stack(ws, 1)  # [B, T]
    T = X.shape[1]
    if not pull:
        # the estimators read the samples as stored, in FP32
        fe = _profile(X.float().double().reshape(lam.size, R, T), torch.from_numpy(lam).cuda(), run.k, run.kT)
        return {"x": X.reshape(-1).cpu().numpy(), "pos": x.cpu().numpy(), "fe": fe}
    m = Wr.amin(0)
    je = m - run.kT * torch.log(torch.exp(-(Wr - m) / run.kT).mean(0))
    mean, var = Wr.mean(0), (Wr - Wr.mean(0)).square().mean(0)
    at = PULL["lambda1"] + PULL["velocity"] * run.dt * run.stride * np.arange(1, T + 1)
    fe = {"dF_JE": je, "dF_cumulant": mean - var / (2 * run.kT), "W_mean": mean, "W_var": var,
          "mean_x": X.float().double().mean(0)}
    return {"x": X.reshape(-1).cpu().numpy(), "work": Wr.cpu().numpy(),
            "fe": {"lambda": at, **{q: t.cpu().numpy() for q, t in fe.items()}}}


def exact(case, seed):
    kind = case["kind"]
    with torch.no_grad():
        if kind == "chain":
            p, start, lam, run = _chain_inputs(case, seed)
            xs, pos = _chain_exact(p, start, lam, run, 0, case["final"])
            return {"x": xs.reshape(-1), **({"pos": pos} if case["final"] else {})}
        if kind == "batch":
            params, starts, lams, run = _batch_inputs(case, seed)
            out, w0 = [], 0
            for p, st, lam in zip(params, starts, lams):
                out.append(_chain_exact(p, st, lam, run, w0 * run.replicas, False)[0].reshape(-1))
                w0 += lam.size
            return {"x": np.concatenate(out)}
        if kind in ("od1d", "pull1d"):
            return _well_exact(case, seed)
        if kind == "reduce":
            x, lam = _store(case, seed)
            return _profile(x.double(), lam, 500.0, KT300)
    return None  # the surrogate's products are BF16: 64 bits is another path of training
