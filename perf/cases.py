"""The work a user of qmcmd has it do, as measurable cases.

Kinds of case (one entry-point sequence each):

* ``md``       one MD step on the device: qmc_energy_forces_device, then
               langevin_step_device with the covariance S it returned (FP64 form).
* ``call``     one energy / force / covariance evaluation on the device
               (qmc_energy_forces_device): the mixed form, which production runs
               use, and the twist-averaged form.
* ``eval``     qmc_eval_config: ln|psi|, E_L and their R-derivatives of given
               configurations, host arrays in and out.
* ``langevin`` one Langevin step on the device with S given, or with the
               empirical S built on the device.
* ``toy``      trajectories of the rotating-spring toy model.
* ``served``   one MD step of each of several trajectories through the server.

Systems are the dense-hydrogen workloads of paper_1605_08423_gb300.synth
(protons, orbital coefficients and start points from the seed).  The handles
come warmed up (their first call, with its longer warm-up, is part of what a
running program has behind it), as walkers carry over from MD step to MD step.

The mixed form evaluates its samples in FP32, so its results are taken as
float32; the FP64 form's are float64.
"""
import math

import numpy as np
import torch

from paper_1605_08423_gb300 import qmcmd as q
from paper_1605_08423_gb300 import synth

ZETA = {1: (0.7,), 2: synth.ZETA_2, 3: (0.4446, 0.727, 1.962), 4: synth.ZETA_4}
ZETA_J = 0.7933844


def _case(name, kind, **kw):
    base = dict(name=name, kind=kind, form="fp64", N=16, G=2, rs=1.4, walkers=256, sweeps=4, recompute=1,
                newton=False, j34=False, twists=0)
    base.update(kw)
    return base


def listed():
    return [
        # the smallest system of the workload table (h16), FP64: a step is many small launches
        _case("md_h16_fp64", "md", N=16, walkers=256, sweeps=20),
        # the paper's 64-atom cell in the reference precision, an inverse recompute every 4 sweeps
        _case("md_h64_fp64", "md", N=64, walkers=1024, sweeps=4, recompute=4),
        # 64 atoms averaged over the 4 x 4 x 4 Monkhorst-Pack mesh of the main text
        _case("twist_h64_fp64", "call", N=64, walkers=512, sweeps=2, recompute=2, twists=64),
        # the production run: 128 atoms, four Gaussians, 16384 walkers, mixed form
        _case("call_h128_mixed", "call", form="mixed", N=128, G=4, rs=1.2, walkers=16384, sweeps=8, recompute=8),
        # 64 atoms in the mixed form with the Newton-Schulz recompute
        _case("call_h64_mixed_newton", "call", form="mixed", N=64, walkers=4096, sweeps=8, recompute=2, newton=True),
        # an uneven cell (27 electrons per spin, three Gaussians, odd walker count) with the paper's
        # production wavefunction (e-e-n-n Jastrow term)
        _case("call_h54_mixed_j34", "call", form="mixed", N=54, G=3, rs=1.3, walkers=1501, sweeps=4, recompute=3,
              j34=True),
        # local energies and derivatives of stored configurations, production size
        _case("eval_h128_mixed", "eval", form="mixed", N=128, G=4, rs=1.2, walkers=1024),
        # the same in FP64 on an uneven cell
        _case("eval_h50_fp64", "eval", N=50, G=4, rs=1.3, walkers=301),
        # the accelerated step alone at the production size (S from elsewhere, e.g. a sharded evaluation)
        _case("langevin_h128_cov", "langevin", N=128, mode="cov"),
        # conventional MD acceleration with the empirical S of the conclusions
        _case("langevin_h108_empirical", "langevin", N=108, mode="empirical"),
        # the SI's integrator comparison
        dict(name="toy_adopted", kind="toy", scheme="adopted", s_mode=0, traj=100003, steps=500),
        # several small trajectories sharing the GPU through the server
        _case("served_h16_h32", "served", N=16, walkers=256, sweeps=4, recompute=2, trajectories=6),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["md", "call", "call", "call", "eval", "eval", "langevin", "toy"])
    rs = round(rng.uniform(1.2, 1.5), 3)
    if kind == "toy":
        return dict(kind="toy", scheme=rng.choice(["adopted", "fast", "first", "standard", "norogna"]), s_mode=0,
                    traj=_log_int(rng, 1000, 200000), steps=_log_int(rng, 50, 500))
    if kind == "langevin":
        c = _case("", kind, N=2 * _log_int(rng, 3, 64), rs=rs, mode=rng.choice(["cov", "cov", "empirical"]))
    elif kind == "md":
        n = _log_int(rng, 3, 32)
        c = _case("", kind, N=2 * n, G=rng.randint(1, 4), rs=rs, walkers=_log_int(rng, 24 * n, 2048),
                  sweeps=rng.randint(1, 6), recompute=rng.randint(1, 4))
    elif kind == "eval":
        form = rng.choice(["fp64", "mixed"])
        n = _log_int(rng, 4, 32 if form == "fp64" else 64)
        c = _case("", kind, form=form, N=2 * n, G=rng.randint(2, 4), rs=rs,
                  walkers=_log_int(rng, 64, 512 if form == "fp64" else 1024), j34=rng.random() < 0.25)
    else:
        if rng.random() < 0.25:
            k = rng.choice([1, 8, 27])
            c = _case("", kind, N=2 * _log_int(rng, 4, 32), rs=rs, walkers=k * rng.randint(8, 19),
                      sweeps=rng.randint(1, 2), recompute=2, twists=k)
        else:
            n = _log_int(rng, 8, 64)
            c = _case("", kind, form="mixed", N=2 * n, G=rng.choice([2, 3, 4]) if n < 64 else 4, rs=rs,
                      walkers=_log_int(rng, 512, 8192), sweeps=rng.randint(1, 8), recompute=rng.randint(1, 8),
                      newton=rng.random() < 0.3, j34=rng.random() < 0.25)
    del c["name"]
    return c


# ---------------------------------------------------------------------------
# Preparation
# ---------------------------------------------------------------------------
def _jastrow(N, seed):
    f = 0.02 * np.random.default_rng(seed + 31).standard_normal((N, N))
    return f + f.T


def _system(c, seed, **over):
    wl = synth.Workload(name=c["kind"], N=c["N"], rs=c["rs"], zeta=ZETA[c["G"]], walkers=c["walkers"],
                        sweeps=c["sweeps"], T_kelvin=1500.0, seed=1000 + seed % 1000003)
    tw = None
    if c["twists"]:
        tw = synth.monkhorst_pack(round(c["twists"] ** (1.0 / 3.0)))
    kw = dict(precision=q.QMC_MIXED if c["form"] == "mixed" else q.QMC_FP64, warmup=8, warmup_cont=1,
              recompute_every=c["recompute"], fj=_jastrow(c["N"], seed) if c["j34"] else None, twists=tw)
    kw.update(over)
    cfg = q.Config.from_workload(wl, **kw)
    return wl, cfg


def _handle(wl, cfg, c):
    s = q.QMCSystem(cfg, wl.R)
    s.set_stream(torch.cuda.current_stream().cuda_stream or 1)
    if c["newton"]:
        s.set_recompute(q.QMC_RECOMPUTE_NEWTON)
    return s


def _dev(a):
    return torch.tensor(np.ascontiguousarray(a, dtype=np.float64), device="cuda")


def _covariance(n3, seed, scale):
    """A positive definite S with eigenvalues over two decades, as a force covariance has."""
    rng = np.random.default_rng(seed)
    Q, _ = np.linalg.qr(rng.standard_normal((n3, n3)))
    return (Q * (scale * 10.0 ** rng.uniform(-1.0, 1.0, n3))) @ Q.T


def _langevin_inputs(c, seed):
    wl = synth.Workload(name="langevin", N=c["N"], rs=c["rs"], zeta=synth.ZETA_2, walkers=2, sweeps=1,
                        seed=1000 + seed % 1000003)
    n3 = 3 * c["N"]
    rng = np.random.default_rng(seed + 5)
    d = dict(wl=wl, R=wl.R.ravel(), f=[0.1 * rng.standard_normal(n3) for _ in range(2)], T=1500.0, delta=0.1, S=None)
    if c["mode"] == "cov":
        d["S"] = [_covariance(n3, seed + k, 1e-3) for k in range(2)]
        d["alpha"] = 40.0
    else:
        d["mu"], d["alpha"] = 12.0, 0.0
    return d


def _configs(c, wl, seed):
    """Electrons scattered around the protons, the better conditioned half of the draws: |psi|^2 sampling
    suppresses configurations near the nodes, where a Slater block is close to singular."""
    W, N, n = c["walkers"], wl.N, wl.N // 2
    X = synth.near_protons(2 * W, wl.R, n, 0.5, wl.L, seed)
    R, C, zeta = _dev(wl.R), _dev(wl.C), _dev(np.array(wl.zeta))
    kappa = []
    for x in torch.split(_dev(X), max(1, int(4.0e7 / (N * N * c["G"])))):
        t = _geometry(x[:, :, None] - R, wl.L)[0]
        A = (torch.exp(-zeta * t[..., None]).reshape(-1, N, N * c["G"]) @ C).reshape(-1, 2, n, n)
        nrm = torch.linalg.matrix_norm
        kappa.append((nrm(A) * nrm(torch.linalg.inv_ex(A)[0])).amax(1))
    return X[torch.argsort(torch.cat(kappa), stable=True)[:W].sort()[0].cpu().numpy()]


def prepare(case, seed):
    c = case
    if c["kind"] == "toy":
        p = q.toy_params(q.TOY_SCHEMES[c["scheme"]], c["s_mode"], n_steps=c["steps"], n_burn=c["steps"] // 5, seed=seed)
        xy = _dev(synth.toy_starts(c["traj"], seed))
        return dict(kind="toy", p=p, xy=xy, out=torch.zeros(c["traj"], q.QMC_TOY_NOUT, dtype=torch.float64, device="cuda"))
    if c["kind"] == "langevin":
        d = _langevin_inputs(c, seed)
        wl = d["wl"]
        s = q.QMCSystem(q.Config.from_workload(wl), wl.R)
        s.set_stream(torch.cuda.current_stream().cuda_stream or 1)
        mode = q.QMC_S_COV if c["mode"] == "cov" else q.QMC_S_EMPIRICAL
        if mode == q.QMC_S_EMPIRICAL:
            s.set_empirical_s(0.0, d["mu"])
        st = dict(kind="langevin", s=s, mode=mode, T=d["T"], delta=d["delta"], alpha=d["alpha"], R=_dev(d["R"]),
                  f=[_dev(f) for f in d["f"]], S=[_dev(S) for S in d["S"]] if d["S"] else [None, None])
        # the step before this one, whose (R, S) the next step's drift term needs
        s.langevin_step_device(st["R"], st["f"][0], st["S"][0], st["T"], st["delta"], mode, st["alpha"])
        s.sync()
        return st
    if c["kind"] == "served":
        srv = q.Server(2 << 30, c["trajectories"])
        tids = []
        for k in range(c["trajectories"]):
            ck = dict(c, N=c["N"] * (1 + k % 2), rs=c["rs"] - 0.05 * (k % 3))
            wl, cfg = _system(ck, seed + 101 * k)
            tids.append(srv.add_trajectory(cfg, wl.R, 1500.0, 0.1))
        st = dict(kind="served", srv=srv, tids=tids)
        run(st)
        return st
    wl, cfg = _system(c, seed)
    s = _handle(wl, cfg, c)
    if c["kind"] == "eval":
        return dict(kind="eval", s=s, X=_configs(c, wl, seed), R=wl.R, mixed=c["form"] == "mixed")
    N = wl.N
    st = dict(kind=c["kind"], s=s, N=N, R=_dev(wl.R), T=wl.T_kelvin, delta=wl.delta, mixed=c["form"] == "mixed",
              out=torch.zeros(4 + 3 * N + 9 * N * N, dtype=torch.float64, device="cuda"))
    s.energy_forces_device(st["R"], st["out"])
    s.sync()
    return st


# ---------------------------------------------------------------------------
# One pass
# ---------------------------------------------------------------------------
def run(st):
    kind = st["kind"]
    if kind == "toy":
        q.toy_langevin_device(st["p"], st["xy"], st["out"], torch.cuda.current_stream().cuda_stream)
        return st["out"]
    if kind == "langevin":
        st["s"].langevin_step_device(st["R"], st["f"][1], st["S"][1], st["T"], st["delta"], st["mode"], st["alpha"])
        return st["R"]
    if kind == "served":
        srv, tids = st["srv"], st["tids"]
        tickets = [srv.submit(t) for t in tids]
        got = {}
        while len(got) < len(tickets):
            srv.progress()
            for tk, tid in zip(tickets, tids):
                if tk not in got:
                    r = srv.fetch(tk, tid)
                    if r is not None:
                        got[tk] = r
        return [{k: got[tk][k] for k in ("status", "E", "E_err", "accept", "f", "S", "R_next")} for tk in tickets]
    if kind == "eval":
        g = st["s"].eval_config(st["X"], st["R"])
        return {k: v.astype(np.float32) for k, v in g.items()} if st["mixed"] else g
    N3, out = 3 * st["N"], st["out"]
    st["s"].energy_forces_device(st["R"], out)
    if kind == "md":
        st["s"].langevin_step_device(st["R"], out[4:4 + N3], out[4 + N3:], st["T"], st["delta"])
    o = out.float() if st["mixed"] else out
    r = dict(E=o[0], E_err=o[1], n_samples=o[2], accept=o[3], f=o[4:4 + N3], S=o[4 + N3:])
    if kind == "md":
        r["R"] = st["R"]
    return r


# ---------------------------------------------------------------------------
# What a pass cannot do without
# ---------------------------------------------------------------------------
def _sample_flops(N, G, j34, z):
    """One E_L and 3N-force sample: derivative rows, K = G Y G, Z and P, pair terms (z = 2: complex orbitals)."""
    n, B = N // 2, N * G
    pairs = 60.0 * (1.5 * N * N) + (16.0 * N ** 3 if j34 else 0.0)
    return z * (2.0 * N * B * n * 4 + 2 * 4.0 * n ** 3 + 2 * 2.0 * N * B * n) + pairs


def _sweep_flops(N, G, z):
    n, B = N // 2, N * G
    return z * (2.0 * N * B * n + N * 4.0 * n * n) + 30.0 * 2 * N * N


def work(case):
    c = case
    if c["kind"] == "toy":
        return dict(bytes=8.0 * 9 * c["traj"], flops=97.0 * c["traj"] * c["steps"])
    N = c["N"]
    N3 = 3 * N
    if c["kind"] == "langevin":
        ns = 2 if c["mode"] == "cov" else 1
        return dict(bytes=8.0 * (ns * N3 * N3 + 4 * N3), flops=N3 ** 3 / 3.0 + 8.0 * N3 * N3)
    W, G, z = c["walkers"], c["G"], 2.0 if c["twists"] else 1.0
    inv = z * 2 * 2.0 * (N // 2) ** 3
    if c["kind"] == "eval":
        return dict(bytes=8.0 * W * (N3 + 2 + 2 * N3) + 8.0 * N3,
                    flops=W * (_sample_flops(N, G, c["j34"], z) + inv + 2.0 * N * N * G * (N // 2)))
    sweeps = c["sweeps"] + 1
    recomputes = 1 + sweeps // c["recompute"]
    flops = W * (c["sweeps"] * _sample_flops(N, G, c["j34"], z) + sweeps * _sweep_flops(N, G, z) +
                 recomputes * (inv + z * 2.0 * N * N * G * (N // 2))) + W * float(N3) * N3
    nbytes = 8.0 * (2 * W * N3 + 4 + N3 + N3 * N3)
    if c["kind"] == "md":
        flops += N3 ** 3 / 3.0
        nbytes += 8.0 * 2 * N3
    if c["kind"] == "served":
        flops *= c["trajectories"] * 3     # half of the trajectories have twice the protons
        nbytes *= c["trajectories"] * 2
    return dict(bytes=nbytes, flops=flops)


# ---------------------------------------------------------------------------
# The same numbers in 64 bits from plain torch / numpy
# ---------------------------------------------------------------------------
_K_B = 3.166811563e-6


def _philox(c0, c1, c2, c3, seed):
    """Philox4x32-10 on int64 tensors holding 32-bit words."""
    m32 = 0xFFFFFFFF
    k0, k1 = seed & m32, (seed >> 32) & m32
    for _ in range(10):
        p0, p1 = c0 * 0xD2511F53, c2 * 0xCD9E8D57
        hi0, lo0 = (p0 >> 32) & m32, p0 & m32
        hi1, lo1 = (p1 >> 32) & m32, p1 & m32
        c0, c1, c2, c3 = hi1 ^ c1 ^ k0, lo1, hi0 ^ c3 ^ k1, lo0
        k0, k1 = (k0 + 0x9E3779B9) & m32, (k1 + 0xBB67AE85) & m32
    return c0, c1, c2, c3


def _u53(a, b):
    return (((a >> 5) << 26 | (b >> 6)).double() + 0.5) / 9007199254740992.0


def _normals(n, step, seed):
    i = torch.arange(n, dtype=torch.int64)
    w = _philox(i, torch.full_like(i, step), torch.zeros_like(i), torch.full_like(i, 7), seed)
    return (torch.sqrt(-2.0 * torch.log(_u53(w[0], w[1]))) * torch.cos(2.0 * math.pi * _u53(w[2], w[3]))).numpy()


def _yukawa_s(R, L, lam, mu):
    N = R.shape[0]
    d = R[:, None] - R[None]
    d -= L * np.rint(d / L)
    H = np.zeros((N, N, 3, 3))
    for c in range(27):
        x = d + L * np.array([c % 3 - 1, (c // 3) % 3 - 1, c // 9 - 1])
        r2 = np.sum(x * x, -1)
        ok = (r2 < L * L) & ~np.eye(N, dtype=bool)
        r2 = np.where(ok, r2, 1.0)
        r = np.sqrt(r2)
        e = np.where(ok, np.exp(-r / lam), 0.0)
        v1 = -e * (1 / r2 + 1 / (lam * r))
        v2 = e * (2 / r ** 3 + 2 / (lam * r2) + 1 / (lam ** 2 * r))
        H += ((v2 - v1 / r) / r2)[..., None, None] * x[..., :, None] * x[..., None, :] + \
            (v1 / r)[..., None, None] * np.eye(3)
    S = -H
    S[np.arange(N), np.arange(N)] = H.sum(1)
    return S.transpose(0, 2, 1, 3).reshape(3 * N, 3 * N) + mu * np.eye(3 * N)


def _exact_langevin(c, seed):
    d = _langevin_inputs(c, seed)
    wl, L, delta, alpha = d["wl"], d["wl"].L, d["delta"], d["alpha"]
    Dt = (1 - math.exp(-alpha * delta)) / alpha if alpha > 0 else delta
    Db = (1 - math.exp(-2 * alpha * delta)) / (2 * alpha) if alpha > 0 else delta
    N = c["N"]
    kF = (3 * math.pi ** 2 * N / L ** 3) ** (1 / 3)
    lam = 1 / math.sqrt(4 * kF / math.pi)
    R = d["R"].copy()
    Rp = Sp = None
    for k in range(2):
        S = d["S"][k] if d["S"] else _yukawa_s(R.reshape(-1, 3), L, lam, d["mu"])
        if Rp is None:
            Rp, Sp = R.copy(), S
        dr = Rp - R
        dr -= L * np.rint(dr / L)
        g = d["f"][k] - (Sp - S) @ dr / (2 * Db)
        low = np.linalg.cholesky(S)
        x = np.linalg.solve(low.T, np.linalg.solve(low, g))
        z = np.linalg.solve(low.T, _normals(3 * N, k, wl.seed))
        Rn = R + Dt * x + math.sqrt(2 * d["T"] * _K_B * Db) * z
        Rp, Sp, R = R, S, Rn - L * np.floor(Rn / L)
    return R


def _exact_toy(c, seed):
    p = q.toy_params(q.TOY_SCHEMES[c["scheme"]], c["s_mode"], n_steps=c["steps"], n_burn=c["steps"] // 5, seed=seed)
    r = _dev(synth.toy_starts(c["traj"], seed)).T.contiguous()
    D, T, k, a = p.delta, p.T, p.k, p.a
    dt = db = D
    if c["scheme"] == "adopted" and p.alpha > 0:
        dt, db = (1 - math.exp(-p.alpha * D)) / p.alpha, (1 - math.exp(-2 * p.alpha * D)) / (2 * p.alpha)
    i = torch.arange(c["traj"], dtype=torch.int64, device="cuda")
    sr = 1.0 / p.lam      # S = P_r / lambda + P_t

    def mul(pr, pt, u, v):  # (pr P_r(u) + pt P_t(u)) v
        rad = (u[0] * v[0] + u[1] * v[1]) / (u[0] ** 2 + u[1] ** 2)
        return (pr - pt) * rad * u + pt * v

    prev, th = r.clone(), torch.zeros_like(r[0])
    su, su2, srr = torch.zeros_like(th), torch.zeros_like(th), torch.zeros_like(th)
    for s in range(c["steps"]):
        w = _philox(i, torch.full_like(i, s), torch.zeros_like(i), torch.full_like(i, 8), seed)
        rho = torch.sqrt(-2.0 * torch.log(_u53(w[0], w[1])))
        ang = 2.0 * math.pi * _u53(w[2], w[3])
        xi = torch.stack([rho * torch.cos(ang), rho * torch.sin(ang)])
        rad = torch.sqrt(r[0] ** 2 + r[1] ** 2)
        f = -k * (rad - a) / rad * r
        sd = (sr - 1.0) / rad ** 2
        s11, s12, s22 = 1 + sd * r[0] ** 2, sd * r[0] * r[1], 1 + sd * r[1] ** 2
        l11 = torch.sqrt(s11)
        l21 = s12 / l11
        l22 = torch.sqrt(s22 - l21 ** 2)
        z1 = xi[1] / l22
        z = torch.stack([(xi[0] - l21 * z1) / l11, z1])
        sf = mul(1 / sr, 1.0, r, f)
        amp = math.sqrt(2 * T * D)
        if c["scheme"] == "standard":
            new = r + D * sf + T * D * (1 / sr - 1.0) / rad ** 2 * r + amp * z
        elif c["scheme"] == "norogna":
            new = r + D * sf + amp * z
        elif c["scheme"] == "first":
            e = amp * z
            y = r + e
            new = y + D * sf - 0.5 * mul(1 / sr, 1.0, r, mul(sr, 1.0, y, e) - mul(sr, 1.0, r, e))
        else:
            e = prev - r
            wv = mul(1 / sr, 1.0, r, mul(sr, 1.0, prev, e) - mul(sr, 1.0, r, e))
            if c["scheme"] == "fast":
                new = r + D * sf + amp * z - 0.5 * wv
            else:
                new = r + dt * (sf - wv / (2 * db)) + math.sqrt(2 * T * db) * z
        th += torch.atan2(r[0] * new[1] - r[1] * new[0], r[0] * new[0] + r[1] * new[1])
        prev, r = r, new
        if s >= c["steps"] // 5:
            rad = torch.sqrt(r[0] ** 2 + r[1] ** 2)
            u = 0.5 * k * (rad - a) ** 2
            su += u
            su2 += u * u
            srr += rad
    return torch.stack([r[0], r[1], su, su2, srr, th, torch.zeros_like(th)], 1)


def _radial(p, qd, f1, f2):
    """Gradient and Laplacian of f(t) from f' and f'' (p, qd: [..., 3])."""
    return 2 * f1[..., None] * p, 4 * f2 * (p * p).sum(-1) + 2 * f1 * qd.sum(-1)


def _geometry(d, L):
    ell = L / math.pi
    s, c = torch.sin(d / ell), torch.cos(d / ell)
    return ell * ell * (s * s).sum(-1), ell * s * c, c * c - s * s


def _ewald_images(d, L, kappa):
    """Sum of erfc(kappa r)/r over the images r < L of each vector's minimum image (zero vectors left out)."""
    d = d - L * torch.round(d.detach() / L)
    v = 0.0
    for c in range(27):
        x = d + L * torch.tensor([c % 3 - 1, (c // 3) % 3 - 1, c // 9 - 1], dtype=d.dtype, device=d.device)
        r2 = (x * x).sum(-1)
        ok = (r2 < L * L) & (r2 > 0)
        r = torch.sqrt(torch.where(ok, r2, torch.ones_like(r2)))
        v = v + torch.where(ok, torch.erfc(kappa * r) / r, torch.zeros_like(r))
    return v


def _exact_eval(c, seed):
    wl, cfg = _system(c, seed)
    N, n, L, kap, b, mmax = wl.N, wl.N // 2, wl.L, wl.kappa, 1.0, cfg.mmax
    X, C, zeta = _dev(_configs(c, wl, seed)), _dev(wl.C), _dev(np.array(wl.zeta))
    fj = _dev(cfg.fj) if c["j34"] else None
    m = np.array([(x, y, z) for x in range(mmax + 1) for y in range(-mmax, mmax + 1) for z in range(-mmax, mmax + 1)
                  if (x > 0 or (x == 0 and y > 0) or (x == 0 and y == 0 and z > 0)) and x * x + y * y + z * z <= mmax * mmax])
    kv = _dev(2 * math.pi / L * m)
    k2 = (kv * kv).sum(-1)
    kw = 4 * math.pi / L ** 3 * torch.exp(-k2 / (4 * kap * kap)) / k2
    off = ~torch.eye(N, dtype=torch.bool, device="cuda")
    upper = torch.triu(torch.ones(N, N, dtype=torch.bool, device="cuda"), 1)
    res = {k: [] for k in ("lnpsi", "el", "dlnpsi", "del_")}
    chunk = max(1, int(2.0e7 / (N * N * c["G"] * 5)))
    for w0 in range(0, c["walkers"], chunk):
        x = X[w0:w0 + chunk]
        W = x.shape[0]
        R = _dev(wl.R)[None].expand(W, N, 3).clone().requires_grad_(True)
        dv = x[:, :, None] - R[:, None]                               # [W, i, a, 3]
        t, p, qd = _geometry(dv, L)
        g, l, lndet = [], [], 0.0
        e = torch.exp(-zeta * t[..., None])                           # [W, i, a, G]
        gr = -2 * zeta * e * 1.0
        lap = 4 * zeta ** 2 * e * (p * p).sum(-1)[..., None] - 2 * zeta * e * qd.sum(-1)[..., None]
        flat = lambda v: v.reshape(W, N, N * c["G"]) @ C              # noqa: E731
        phi, lp = flat(e), flat(lap)
        D = torch.stack([flat(gr * p[..., mu, None]) for mu in range(3)], -1)   # [W, i, j, 3]
        for sp in range(2):
            rows = slice(sp * n, sp * n + n)
            inv = torch.linalg.inv(phi[:, rows])                      # [W, j, i]
            lndet = lndet + torch.linalg.slogdet(phi[:, rows])[1]
            g.append(torch.einsum("wijm,wji->wim", D[:, rows], inv))
            l.append(torch.einsum("wij,wji->wi", lp[:, rows], inv))
        g, l = torch.cat(g, 1), torch.cat(l, 1)
        # Pade e-n and e-e terms
        rho = torch.sqrt(t)
        iq = 1 / (1 + b * rho)
        u1, u2 = -iq ** 2, 2 * b * iq ** 3
        U = (-rho * iq).sum((1, 2))
        gu, lu = _radial(p, qd, 0.5 * u1 / rho, 0.25 * (u2 / rho ** 2 - u1 / rho ** 3))
        gu, lu = gu.sum(2), lu.sum(2)
        te, pe, qe = _geometry(x[:, :, None] - x[:, None], L)
        re = torch.sqrt(torch.where(off, te, torch.ones_like(te)))
        iq = 1 / (1 + b * re)
        u1, u2 = 0.5 * iq ** 2, -b * iq ** 3
        ge, le = _radial(pe, qe, 0.5 * u1 / re, 0.25 * (u2 / re ** 2 - u1 / re ** 3))
        gu = gu + torch.where(off[..., None], ge, 0.0).sum(2)
        lu = lu + torch.where(off, le, 0.0).sum(2)
        U = U + torch.where(upper, 0.5 * re * iq, 0.0).sum((1, 2))
        if fj is not None:
            ch = torch.exp(-ZETA_J * t)                               # [W, i, a]
            gch, lch = _radial(p, qd, -ZETA_J * ch, ZETA_J ** 2 * ch)
            wv = (ch.sum(1, keepdim=True) - ch) @ fj
            U = U + 0.5 * (ch * wv).sum((1, 2))
            gu = gu + (gch * wv[..., None]).sum(2)
            lu = lu + (lch * wv).sum(2)
        kin = (l - (g * g).sum(-1) + lu + ((g + gu) ** 2).sum(-1)).sum(1)
        # Ewald: electrons -1, protons +1
        pp = R[:, :, None] - R[:, None]
        pp = torch.where(off[..., None], pp, 0.0)
        ee = torch.where(off[..., None], x[:, :, None] - x[:, None], 0.0)
        one = torch.where(off, 1.0, 0.0).double()
        real = 0.5 * (_ewald_images(pp, L, kap) * one).sum((1, 2)) + 0.5 * (_ewald_images(ee, L, kap) * one).sum((1, 2)) \
            - _ewald_images(dv, L, kap).sum((1, 2))
        pa, pb = R @ kv.T, x @ kv.T
        rec = (kw * ((torch.cos(pa).sum(1) - torch.cos(pb).sum(1)) ** 2 +
                     (torch.sin(pa).sum(1) - torch.sin(pb).sum(1)) ** 2)).sum(-1)
        el = -0.5 * kin + real + rec - kap / math.sqrt(math.pi) * 2 * N
        lnpsi = lndet + U
        d1, = torch.autograd.grad(lnpsi.sum(), R, retain_graph=True)
        d2, = torch.autograd.grad(el.sum(), R)
        for key, v in zip(("lnpsi", "el", "dlnpsi", "del_"), (lnpsi, el, d1, d2)):
            res[key].append(v.detach())
    return {k: torch.cat(v).cpu().numpy() for k, v in res.items()}


def exact(case, seed):
    if case["kind"] == "eval":
        return _exact_eval(case, seed)
    if case["kind"] == "langevin":
        return _exact_langevin(case, seed)
    if case["kind"] == "toy":
        return _exact_toy(case, seed)
    return None     # a Markov chain: its samples have no value but the chain's own
