"""What users of this framework run, as measurable cases.

Each case is one call (or one short sequence of calls) of the public Python
API: ground-state solves, Schwarz iterations of real-time and batched
problems, training-set generation and training of the learned initial traces,
and the local-determinant builder.  `listed()` gives the named cases, `draw()`
more of the same ranges; `prepare()` makes what a program holds before the
call, `run()` is the call, `exact()` restates its outputs in plain 64-bit
torch / numpy.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_1710_02401_gb300 import learn
from paper_1710_02401_gb300 import problems as P
from paper_1710_02401_gb300 import swr as S

DEVICE = "cuda:0"
TOL = 1e-8  # interface residual at which a solve counts as converged
PRECISIONS = {"fp64": S.PREC_FP64, "mixed": S.PREC_MIXED, "refined": S.PREC_FP32_REFINED}


# ---------------------------------------------------------------- the cases

def _ground(name, n_elec, half, L, overlap, K_d, q_p, precision, kmax, delta=0.0, eta=0.5, anti=False):
    return {"kind": "ground", "n_elec": n_elec, "half": half, "L": L, "overlap": overlap, "K_d": K_d, "q_p": q_p,
            "delta": delta, "eta": eta, "precision": precision, "kmax": kmax, "anti": anti,
            **({"name": name} if name else {})}


def _time(name, half, L, overlap, K_d, q_p, n_steps, precision, n_elec=2):
    return {"kind": "time", "n_elec": n_elec, "half": half, "L": L, "overlap": overlap, "K_d": K_d, "q_p": q_p,
            "n_steps": n_steps, "precision": precision, **({"name": name} if name else {})}


def listed():
    return [
        # the smallest solve in earnest use: one electron, two subdomains, the
        # default precision; a window step is a few microseconds of work, so
        # latency is all there is
        _ground("ground_1e_2sd_fp64", 1, 10.0, 2, 1.0, 40, 14, "fp64", 6, delta=4.0, eta=1.0),
        # an exploratory two-electron run: nine small subdomains, odd sizes
        _ground("ground_2e_9sd_mixed", 2, 6.0, 3, 0.4, 11, 8, "mixed", 6),
        # the headline ground-state workload (16 subdomains, 24 x 24 Gaussians),
        # assembly and the first Schwarz iterations of its solve
        _ground("ground_2e_16sd_mixed", 2, 12.0, 4, 0.6, 24, 12, "mixed", 8),
        # the same problem on the plain FP64 path, the default of the API
        _ground("ground_2e_16sd_fp64", 2, 12.0, 4, 0.6, 24, 12, "fp64", 3),
        # the lowest antisymmetric (triplet) state of the same problem
        _ground("triplet_2e_16sd_mixed", 2, 12.0, 4, 0.6, 24, 12, "mixed", 3, anti=True),
        # a parameter study: independent one- and two-electron problems with
        # uneven bases in one context, one Schwarz iteration of all of them
        {"name": "batch_32_uneven_mixed", "kind": "batch", "instances": 32, "n_steps": 200, "precision": "mixed"},
        # the real-time workload (64 subdomains, 32 x 32 Gaussians, dipole pulse),
        # one Schwarz iteration over a quarter of its 1000 steps
        _time("real_time_64sd_mixed", 20.0, 8, 0.5, 32, 14, 250, "mixed"),
        # the same in plain FP64, a shorter window
        _time("real_time_64sd_fp64", 20.0, 8, 0.5, 32, 14, 100, "fp64"),
        # a training set for the learned initial traces: a batch of small
        # real-time problems solved a few iterations and encoded
        {"name": "trace_training_set", "kind": "traces", "instances": 12, "kmax": 3},
        # one Adam step of the trace predictor on a whole training set
        {"name": "mlp_train_2560", "kind": "mlp_train", "batch": 2560, "width": 256, "hidden": 3},
        # prediction of the initial traces of one 16-subdomain problem
        {"name": "mlp_predict_16", "kind": "mlp_predict", "batch": 16, "width": 256, "hidden": 3},
        # local orbitals and Slater determinants at the paper's Test 1 sizes
        {"name": "determinants_test1", "kind": "lsd", "L": 5, "M": 10, "K": 45, "kd": 40, "q_p": 12, "panel": 0.2},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("ground", "ground", "ground", "time", "time", "batch", "traces", "mlp_train", "mlp_predict",
                       "lsd"))
    if kind == "ground" and rng.random() < 0.35:
        return _ground(None, 1, 10.0, rng.randint(2, 12), round(rng.uniform(0.4, 1.2), 3), rng.randint(12, 44),
                       rng.randint(10, 16), rng.choice(("fp64", "mixed")), rng.randint(2, 6), eta=1.0)
    if kind == "ground":
        L, prec, anti = rng.randint(2, 5), rng.choice(("mixed", "mixed", "fp64", "refined")), rng.random() < 0.2
        kd = rng.randint(8, 24 if L <= 4 else 18)
        return _ground(None, 2, round(2.0 * L + rng.uniform(0.0, L), 2), L, round(rng.uniform(0.35, 0.6), 3), kd,
                       rng.randint(9, 12), prec, rng.randint(2, 3), anti=anti)
    if kind == "time":
        L = rng.randint(2, 8)
        return _time(None, 2.5 * L, L, 0.5, _log(rng, 6, 32), rng.randint(11, 14), _log(rng, 20, 100),
                     rng.choice(("mixed", "mixed", "fp64")))
    if kind == "batch":
        return {"kind": "batch", "instances": _log(rng, 3, 32), "n_steps": rng.randint(60, 190),
                "precision": rng.choice(("mixed", "mixed", "fp64"))}
    if kind == "traces":
        return {"kind": "traces", "instances": rng.randint(2, 11), "kmax": rng.randint(2, 3)}
    if kind == "mlp_train":
        return {"kind": "mlp_train", "batch": _log(rng, 100, 2500), "width": rng.choice((128, 192, 256)),
                "hidden": rng.randint(2, 3)}
    if kind == "mlp_predict":
        return {"kind": "mlp_predict", "batch": _log(rng, 4, 2500), "width": rng.choice((128, 192, 256)),
                "hidden": rng.randint(2, 3)}
    M = rng.randint(5, 10)
    return {"kind": "lsd", "L": rng.randint(3, 5), "M": M, "K": rng.randint(M, M * (M - 1) // 2),
            "kd": 2 * rng.randint(12, 20), "q_p": rng.randint(10, 12), "panel": 0.2}


# ------------------------------------------------------------------- inputs

def _instance(c, seed):
    """The problem of a single-instance case: a molecule whose nuclei and
    softening vary with the seed."""
    rng = random.Random(1000003 * seed + 17)
    box, two, real = (-c["half"], c["half"]), c["n_elec"] == 2, c["kind"] == "time"
    kw = dict(n_elec=c["n_elec"], box=box, L=c["L"], overlap=c["overlap"], K_d=c["K_d"], q_p=c["q_p"],
              delta=c.get("delta") or P.spacing_rule_delta(box, c["L"], c["overlap"], c["K_d"]),
              n_mid=P.mid_panels(box, c["L"], c["overlap"]), ee_coef=1.0 if two else 0.0, eta_ee=0.5,
              eta_en=c.get("eta", 0.5) * rng.uniform(0.95, 1.05), phi0_gamma=1.0)
    d = rng.uniform(0.6, 0.8)
    kw["nuclei"] = ((-d, 1.0), (d, 1.0)) if two else ((rng.uniform(-0.1, 0.1), 1.0),)
    if c["n_elec"] == 1 and c.get("delta"):
        kw["n_mid"] = 9
    if real:
        kw.update(mode=P.TDSE, mu=-10j, dt=0.01, n_steps=c["n_steps"], field=(0.05, 10.0, 0.057, rng.uniform(0, 0.1)),
                  phi0_center=(0.5, 0.3))
    else:
        kw.update(mode=P.TISE, mu=10.0, dt=0.1, ngf_tol=1e-12, max_steps=5000)
        if c["anti"]:
            kw.update(symmetry="antisymmetric", phi0_center=(0.8, -0.8))
    return P.Instance(**kw)


def _batch(c, seed):
    """The seeded uneven batch with a fixed window; geometry and bases are the
    family's, the molecules vary with the seed."""
    rng, out = random.Random(1000003 * seed + 23), []
    for i in P.batched_uneven(c["instances"]):
        eps = rng.uniform(0.3, 1.0)
        out.append(i.replace(ngf_tol=0.0, n_steps=c["n_steps"], eta_en=eps, eta_ee=eps,
                             nuclei=tuple((rng.uniform(-2.0, 2.0), z) for _, z in i.nuclei)))
    return out


def _mlp_dims(c):
    return [learn.N_FEATURES] + [c["width"]] * c["hidden"] + [8 * learn.CODE_S * learn.CODE_T]


def _mlp_inputs(c, seed):
    """Descriptors of seeded subdomains, standardised targets, initial weights."""
    n = -(-c["batch"] // 16)
    x = learn.descriptors(P.learned_trace_family_16sd(n, seed))[:c["batch"]]
    t = np.random.default_rng(seed).standard_normal((c["batch"], _mlp_dims(c)[-1])).astype(np.float32)
    return x, t, learn.init_params(_mlp_dims(c), seed)


def _lsd_args(c, seed):
    rng = random.Random(1000003 * seed + 29)
    return dict(L=c["L"], M=c["M"], K=c["K"], kd=c["kd"], q_p=c["q_p"], panel=c["panel"],
                nuclei=((-rng.uniform(0.4, 0.6), 1.0), (rng.uniform(0.4, 0.6), 1.0)))


def prepare(case, seed):
    c = dict(case)
    kind = c["kind"]
    if kind in ("ground", "time", "batch"):
        insts = _batch(c, seed) if kind == "batch" else [_instance(c, seed)]
        s = S.SWR(insts, precision=PRECISIONS[c["precision"]], device=DEVICE)
        if kind != "ground":
            s.assemble()
        return {"case": c, "swr": s}
    if kind == "traces":
        return {"case": c, "instances": P.learned_trace_family_16sd(c["instances"], seed)}
    if kind in ("mlp_train", "mlp_predict"):
        x, t, p = _mlp_inputs(c, seed)
        mlp = S.MLP(learn.N_FEATURES, c["width"], c["hidden"], _mlp_dims(c)[-1], device=DEVICE)
        mlp.set_params(p)
        return {"case": c, "mlp": mlp, "x": torch.as_tensor(x, device=DEVICE), "t": torch.as_tensor(t, device=DEVICE)}
    return {"case": c, "args": _lsd_args(c, seed)}


# ------------------------------------------------------------------ the call

def run(state):
    c = state["case"]
    kind = c["kind"]
    if kind == "ground":    # a solve: assembly and Schwarz iterations, then the state and its energy
        s = state["swr"]
        s.assemble()
        s.iterate(TOL, c["kmax"])
        return {"energy": s.energy(), "psi": s.get(S.FIELD_PSI_NODES)}
    if kind == "time":      # one Schwarz iteration of a real-time problem
        s = state["swr"]
        rep = s.step()
        return {"res": rep.res, "norm2": s.norm2(), "dipole": s.dipole(), "psi": s.get(S.FIELD_PSI_NODES)}
    if kind == "batch":     # one Schwarz iteration of every instance
        s = state["swr"]
        s.step()
        return {"res": s.residual(), "energy": s.energy(), "psi": s.get(S.FIELD_PSI_NODES)}
    if kind == "traces":
        x, codes, done = learn.gather_training_set(state["instances"], tol=TOL, kmax=c["kmax"])
        return {"x": x, "codes": codes, "done": done}
    if kind == "mlp_train":
        loss, grad = state["mlp"].train_step(state["x"], state["t"], 1e-3, want_grad=True)
        return {"loss": loss, "grad": grad}
    if kind == "mlp_predict":
        return {"y": state["mlp"].forward(state["x"])}
    return S.lsd_build(**state["args"])


# ------------------------------------------------------------------- the work

def _swr_work(insts, steps, elem, sweeps, assemble):
    """Bytes and FP64-equivalent flops of `steps` steps of every subdomain:
    each step applies every step matrix once per sweep; matrices that fit the
    chip's caches are read once, larger sets once per step."""
    mats = flops = psi = inv = 0.0
    for i in insts:
        for s in range(i.n_sub):
            K = float(i.k_d_of(s) ** i.n_elec)
            mats += elem * K * K
            flops += (elem // 8) ** 2 * 2.0 * K * K * sweeps * steps
            inv += 2.0 * K ** 3
            psi += 8.0 * (elem // 8) * float((i.n_mid + 2) * i.q_p) ** i.n_elec
    reads = steps if mats > 126e6 else 1
    return {"bytes": mats * reads + psi, "flops": flops + (inv if assemble else 0.0)}


def work(case):
    kind = case["kind"]
    if kind == "ground":  # windows of about 500 steps
        return _swr_work([_instance(case, 0)], 500 * case["kmax"], 8, 1, True)
    if kind == "time":
        return _swr_work([_instance(case, 0)], case["n_steps"], 16, 4, False)
    if kind == "batch":
        return _swr_work(_batch(case, 0), case["n_steps"], 8, 1, False)
    if kind == "traces":
        insts = P.learned_trace_family_16sd(case["instances"], 0)
        return _swr_work(insts, 100 * case["kmax"], 16, 6, True)
    if kind in ("mlp_train", "mlp_predict"):
        d, b = _mlp_dims(case), case["batch"]
        mac = float(sum(m * n for m, n in zip(d[:-1], d[1:])))
        if kind == "mlp_predict":
            return {"bytes": 4.0 * (mac + b * (d[0] + d[-1])), "flops": 2.0 * b * mac}
        return {"bytes": 4.0 * (8.0 * mac + b * (d[0] + d[-1])), "flops": 6.0 * b * mac}
    LM, q = case["L"] * case["M"], 16.0 / case["panel"] * case["q_p"]
    M2 = 4.0 * case["M"] ** 2
    return {"bytes": 8.0 * (3 * LM * LM + 3 * case["L"] ** 2 * case["K"] ** 2),
            "flops": case["L"] ** 2 * (2.0 * M2 * q * q + 2.0 * M2 * M2 * q)}


# ---------------------------------------------------- plain 64-bit restatement

def _np_rule(breaks, q):
    t, w = np.polynomial.legendre.leggauss(q)
    p0, p1 = np.asarray(breaks[:-1])[:, None], np.asarray(breaks[1:])[:, None]
    return (0.5 * (p1 - p0) * t + 0.5 * (p1 + p0)).ravel(), (0.5 * (p1 - p0) * w + 0.0 * t).ravel()


class _Line:
    """One coordinate of one subdomain: quadrature, orthonormalised Gaussians
    and their 1-D matrices."""

    def __init__(self, inst, k, kd, delta):
        a, b = inst.box
        H, e, m = (b - a) / inst.L, inst.overlap, inst.n_mid
        self.lo, self.hi, self.k = a + k * H - 0.5 * e, a + (k + 1) * H + 0.5 * e, k
        lo, hi = self.lo, self.hi
        self.x, self.w = _np_rule([lo] + [lo + e + (hi - lo - 2 * e) * j / m for j in range(m)] + [hi - e, hi], inst.q_p)
        chi = np.ones_like(self.x)
        if k > 0:
            chi[:inst.q_p] = 0.5
        if k < inst.L - 1:
            chi[-inst.q_p:] = 0.5
        self.wc = self.w * chi
        self.cen, self.delta, self.X = np.linspace(lo, hi, kd), delta, np.eye(kd)
        v = 0.5 * inst.harmonic * self.x ** 2
        for xa, za in inst.nuclei:
            v = v - za / np.sqrt((self.x - xa) ** 2 + inst.eta_en ** 2)
        B = self.val(self.x)
        self.X = np.linalg.inv(np.linalg.cholesky(B.T @ (self.w[:, None] * B))).T
        self.B, self.D, self.v = self.val(self.x), self.der(self.x), v
        self.T = self.D.T @ (self.w[:, None] * self.D)
        self.U = self.B.T @ ((self.w * v)[:, None] * self.B)
        self.Q = self.B.T @ ((self.w * self.x)[:, None] * self.B)
        self.C = self.B.T @ (self.wc[:, None] * self.B)
        self.R = np.zeros((kd, kd))
        for pos, inner in ((lo, k > 0), (hi, k < inst.L - 1)):
            if inner:
                l = self.val(np.array([pos]))
                self.R += l.T @ l

    def val(self, x):
        return np.exp(-self.delta * (x[:, None] - self.cen) ** 2) @ self.X

    def der(self, x):
        r = x[:, None] - self.cen
        return (-2.0 * self.delta * r * np.exp(-self.delta * r * r)) @ self.X


def _exact_swr(inst, kmax, tol, dev, want_codes=None):
    """kmax Schwarz iterations (or until Res <= tol) of one instance in 64
    bits.  Vectors are [sub][b][a], zero-padded to the largest basis."""
    f, N, L, nsub = torch.float64, inst.n_elec, inst.L, inst.n_sub
    real = inst.mode == P.TDSE
    ty = torch.complex128 if real else f
    up = lambda v, t=f: torch.as_tensor(np.ascontiguousarray(v), dtype=t, device=dev)  # noqa: E731
    kds = [inst.k_d_of(s) for s in range(nsub)]
    km = max(kds)
    kb = km if N == 2 else 1
    lines = [[_Line(inst, (s // L ** d) % L, kds[s], inst.delta_of(s)) for d in range(N)] for s in range(nsub)]
    one = np.ones((1, 1))
    pad = lambda M, n: np.pad(M, ((0, n - M.shape[0]), (0, n - M.shape[1])))  # noqa: E731
    C1 = up(np.stack([pad(l[0].C, km) for l in lines]), ty)
    C2 = up(np.stack([pad(l[1].C if N == 2 else one, kb) for l in lines]), ty)
    Q1 = up(np.stack([pad(l[0].Q, km) for l in lines]), ty)
    Q2 = up(np.stack([pad(l[1].Q if N == 2 else 0 * one, kb) for l in lines]), ty)
    kap, dt, mu = inst.kinetic, inst.dt, complex(inst.mu)
    G = torch.zeros(nsub, kb * km, kb * km, dtype=ty, device=dev)
    c0 = torch.zeros(nsub, kb, km, dtype=ty, device=dev)
    for s, l in enumerate(lines):
        kd = kds[s]
        k2 = kd if N == 2 else 1
        h = [kap * (e.T + mu * e.R) + e.U for e in l]
        H = up(np.kron(np.eye(k2), h[0]), torch.complex128)
        g = [e.B.T @ (e.w * np.exp(-inst.phi0_gamma * (e.x - inst.phi0_center[d]) ** 2)) for d, e in enumerate(l)]
        if N == 2:
            H = H + up(np.kron(h[1], np.eye(kd)), torch.complex128)
            if inst.ee_coef:
                W = up(inst.ee_coef * l[0].w[:, None] * l[1].w / np.sqrt((l[0].x[:, None] - l[1].x) ** 2 + inst.eta_ee ** 2))
                P1, P2 = ((up(e.B)[:, :, None] * up(e.B)[:, None, :]).reshape(-1, kd * kd) for e in l)
                V = (P1.T @ (W @ P2)).reshape(kd, kd, kd, kd).permute(2, 0, 3, 1)  # [b, a, e, c]
                H = H + V.reshape(kd * kd, kd * kd)
        M = torch.eye(k2 * kd, dtype=ty, device=dev) + (0.5j * dt * H if real else dt * H.real)
        Gp = torch.zeros(kb, km, kb, km, dtype=ty, device=dev)
        Gp[:k2, :kd, :k2, :kd] = torch.linalg.inv(M).reshape(k2, kd, k2, kd)
        G[s] = Gp.reshape(kb * km, kb * km)
        c0[s, :k2, :kd] = up(np.outer(g[1] if N == 2 else [1.0], g[0]), ty)

    def norm2(y):
        return (y.conj() * (C2 @ y @ C1)).sum().real

    anti = inst.symmetry == "antisymmetric"
    mir = torch.as_tensor([s // L + L * (s % L) if N == 2 else s for s in range(nsub)], device=dev)

    def proj(y):
        return 0.5 * (y - y[mir].transpose(1, 2)) if anti else y

    c0 = proj(c0)
    if not real and inst.normalize:
        c0 = c0 / norm2(c0).sqrt()

    # interface operators: own values and the averaged Robin data of each subdomain
    def rows(e, d_val, tang_val, j):
        """[points][b][a] of basis j from its factors along the edge's normal and tangent."""
        if N == 1:
            return d_val[:, None, :]
        a, b = (d_val, tang_val) if e == 0 else (tang_val, d_val)
        return b[:, :, None] * a[:, None, :]

    def padrows(r):
        return np.pad(r, ((0, 0), (0, kb - r.shape[1]), (0, km - r.shape[2]))).reshape(r.shape[0], -1)

    own, gw, rob, slots = [], [], [], []
    for s, l in enumerate(lines):
        o, w, per, sl = [], [], {}, []
        for d in range(N):
            for sg, pos, inner in ((-1.0, l[d].lo, l[d].k > 0), (1.0, l[d].hi, l[d].k < L - 1)):
                if not inner:
                    continue
                t = l[1 - d].x if N == 2 else np.zeros(1)
                at, p1 = sum(len(v) for v in w), np.array([pos])
                o.append(padrows(rows(d, np.repeat(l[d].val(p1), t.size, 0), l[1 - d].val(t) if N == 2 else None, s)))
                w.append(l[1 - d].w if N == 2 else np.ones(1))
                sl.append((2 * d + (sg > 0), at, t.size))
                for jd in (l[d].k, l[d].k + int(sg)):
                    for jo in (range(L) if N == 2 else (0,)):
                        j = (jd + L * jo if d == 0 else jo + L * jd) if N == 2 else jd
                        if j == s:
                            continue
                        lj = lines[j]
                        m = np.nonzero((lj[1 - d].lo <= t) & (t <= lj[1 - d].hi))[0] if N == 2 else np.array([0])
                        if not m.size:
                            continue
                        tv = lj[1 - d].val(t[m]) if N == 2 else None
                        val = padrows(rows(d, np.repeat(lj[d].val(p1), m.size, 0), tv, j))
                        der = padrows(rows(d, np.repeat(lj[d].der(p1), m.size, 0), tv, j))
                        r = (mu if real else mu.real) * val + (sg * der if inst.tc != "dirichlet" else 0.0)
                        per.setdefault(j, []).append((at + m, r))
        own.append(up(np.concatenate(o) if o else np.zeros((0, kb * km)), ty))
        gw.append(up(np.concatenate(w) if w else np.zeros(0)))
        n = gw[-1].numel()
        cnt = np.zeros(n)
        for pieces in per.values():
            for at, _ in pieces:
                cnt[at] += 1
        rob.append([])
        if kmax > 1 or want_codes:
            for j, pieces in per.items():
                D = np.zeros((n, kb * km), dtype=complex if real else float)
                for at, r in pieces:
                    D[at] += r / cnt[at][:, None]
                rob[-1].append((j, up(D, ty)))
        slots.append(sl)

    def field(t):
        E0, T, om, ph = inst.field
        return 0.0 if E0 == 0.0 or t < 0 or t > T else E0 * math.sin(math.pi * t / T) ** 2 * math.sin(om * t + ph)

    fixed = inst.window()
    b_prev, u_prev, res = None, None, []
    gemv = lambda y: torch.bmm(G, y.reshape(nsub, -1, 1)).reshape(nsub, kb, km)  # noqa: E731
    Qx = lambda y: y @ Q1.transpose(1, 2) + Q2 @ y  # noqa: E731
    for k in range(kmax):
        c, raw, hist = c0, [c0], [c0]
        wp = 0 if b_prev is None else b_prev.shape[0] - 1
        for n in range(fixed if fixed > 0 else inst.max_steps):
            if real:
                t0, t1 = 0.5 * dt * field(n * dt), 0.5 * dt * field((n + 1) * dt)
                r = 2.0 * c + 1j * (t1 - t0) * Qx(c)
                if wp:
                    r = r + 0.5j * dt * kap * (b_prev[min(n + 1, wp)] + b_prev[min(n, wp)])
                x = gemv(r)
                rho = abs(t1) * N * max(abs(inst.box[0]), abs(inst.box[1]), 1e-3) * 1.05
                for _ in range(0 if rho == 0 else int(math.ceil(math.log(1e-17) / math.log(rho)))):
                    x = gemv(r - 1j * t1 * Qx(x))
                new = y = x - c
            else:
                y = proj(c) if anti else c
                if wp:
                    b = b_prev[min(n + 1, wp)]
                    y = y + kap * dt * (proj(b) if anti else b)
                y = gemv(y)
                new = y / norm2(y).sqrt() if inst.normalize else y
            raw.append(y)
            hist.append(new)
            d, c = new - c, new
            if not real and fixed == 0 and float(norm2(d)) <= inst.ngf_tol ** 2:
                break
        Y, Cn = torch.stack(raw), torch.stack(hist)
        u = [Cn[:, s].reshape(len(hist), -1) @ own[s].T for s in range(nsub)]
        last = u_prev[0].shape[0] if u_prev else 1
        span, r2 = max(len(hist), last) - 1, 0.0
        for s in range(nsub):
            idx = torch.arange(1, span + 1, device=dev)
            a = u[s][idx.clamp(max=len(hist) - 1)]
            if u_prev:
                a = a - u_prev[s][idx.clamp(max=last - 1)]
            r2 = r2 + dt * (gw[s] * a.abs() ** 2).sum()
        res.append(float(torch.as_tensor(r2).sqrt()))
        if kmax > 1 or want_codes:
            g = [sum(Y[:, j].reshape(len(raw), -1) @ D.T for j, D in rob[s]) if rob[s] else None for s in range(nsub)]
            b_prev = torch.stack([((g[s] * gw[s]) @ own[s]).reshape(len(raw), kb, km) if rob[s] else
                                  torch.zeros_like(Y[:, s]) for s in range(nsub)], dim=1)
        u_prev = u
        if res[-1] <= tol:
            break
    num = den = dip = 0.0
    psi = []
    for s, l in enumerate(lines):
        kd = kds[s]
        y = c[s, :kd if N == 2 else 1, :kd]
        B1, D1 = up(l[0].B, ty), up(l[0].D, ty)
        B2, D2 = (up(l[1].B, ty), up(l[1].D, ty)) if N == 2 else (up(one, ty), up(0 * one, ty))
        p, d1, d2 = B2 @ y @ B1.T, B2 @ y @ D1.T, D2 @ y @ B1.T
        x1, x2 = up(l[0].x)[None, :], up(l[1].x)[:, None] if N == 2 else torch.zeros(1, 1, dtype=f, device=dev)
        V = up(l[0].v)[None, :] + (up(l[1].v)[:, None] if N == 2 else 0.0)
        if N == 2 and inst.ee_coef:
            V = V + inst.ee_coef / ((x1 - x2) ** 2 + inst.eta_ee ** 2).sqrt()
        wc = up(l[0].wc)[None, :] * (up(l[1].wc)[:, None] if N == 2 else 1.0)
        num += (wc * (kap * (d1.abs() ** 2 + d2.abs() ** 2) + V * p.abs() ** 2)).sum()
        den += (wc * p.abs() ** 2).sum()
        dip += (wc * (x1 + x2) * p.abs() ** 2).sum()
        psi.append((torch.view_as_real(p.reshape(-1)) if real else p).reshape(-1).cpu().numpy())
    out = {"res": res, "energy": float(num / den), "norm2": float(den), "dipole": float(dip / den),
           "psi": np.concatenate(psi)}
    if want_codes:
        S_, T_ = want_codes
        W = len(raw) - 1

        def ortho(x, w, n):
            M = np.polynomial.chebyshev.chebvander(x, n - 1)
            for q in range(n):
                for _ in range(2):
                    M[:, q] -= M[:, :q] @ (M[:, :q].T @ (w * M[:, q]))
                M[:, q] /= math.sqrt((w * M[:, q] ** 2).sum())
            return M

        Psi = ortho(2.0 * np.arange(W + 1) / W - 1.0, np.ones(W + 1), T_)
        code = np.zeros((nsub, 4, 2, S_, T_))
        for s, l in enumerate(lines):
            for slot, at, m in slots[s]:
                e = l[1 - slot // 2]
                Phi = ortho(2.0 * (e.x - e.lo) / (e.hi - e.lo) - 1.0, e.w, S_)
                gg = g[s][:, at:at + m].cpu().numpy()
                pr = Phi.T @ (e.w[:, None] * gg.T) @ Psi
                code[s, slot, 0], code[s, slot, 1] = pr.real, pr.imag
        out["codes"] = code.reshape(nsub, -1)
    return out


def _exact_mlp(c, seed, train, dev):
    x, t, p = _mlp_inputs(c, seed)
    d = _mlp_dims(c)
    f = lambda a: torch.as_tensor(a, dtype=torch.float64, device=dev)  # noqa: E731
    p = f(p).requires_grad_(train)
    h, o = f(x), 0
    for l, (m, n) in enumerate(zip(d[:-1], d[1:])):
        h = h @ p[o:o + m * n].reshape(m, n) + p[o + m * n:o + m * n + n]
        o += m * n + n
        h = torch.tanh(h) if l < len(d) - 2 else h
    if not train:
        return {"y": h}
    loss = ((h - f(t)) ** 2).mean()
    loss.backward()
    return {"loss": float(loss), "grad": p.grad}


def _exact_lsd(a):
    """Orbitals by Cholesky-reduced symmetric eigenproblems, integrals by the
    same composite rules; the call's remaining arguments at their defaults."""
    lo, hi, ov, eta, eps_b, v_inf = -8.0, 8.0, 0.32, 0.5, 0.4, 100.0
    L, M, K, kd, q, pan = a["L"], a["M"], a["K"], a["kd"], a["q_p"], a["panel"]
    H = (hi - lo) / L
    xb = 0.5 * (H + ov)
    delta = 0.5 / (2.0 * xb / (kd - 1)) ** 2
    margin = max(eps_b, 8.0 / math.sqrt(2.0 * delta))

    def rule(p0, p1, breaks=()):
        pts = sorted({p0, p1, *[b for b in breaks if p0 < b < p1]})
        br = [pts[0]]
        for u, v in zip(pts[:-1], pts[1:]):
            n = max(1, int(math.ceil((v - u) / pan)))
            br += [u + (v - u) * (k + 1) / n for k in range(n)]
        return _np_rule(br, q)

    def ven(x):
        return sum(-z / np.sqrt((x - xa) ** 2 + eta ** 2) for xa, z in a["nuclei"])

    def table(cen, x):
        r = x - cen[:, None]
        g = np.exp(-delta * r * r)
        return g, -2.0 * delta * r * g

    xg, wg = rule(lo - 0.5 * ov - margin, hi + 0.5 * ov + margin)
    lam, coef, F, dF = [], [], [], []
    for i in range(L):
        xc = lo + (i + 0.5) * H
        cen = np.linspace(xc - xb, xc + xb, kd)
        br = [xc - xb - eps_b / 2, xc - xb + eps_b / 2, xc + xb - eps_b / 2, xc + xb + eps_b / 2]
        x, w = rule(xc - xb - margin, xc + xb + margin, br)
        g, dg = table(cen, x)
        u = np.clip((np.abs(x - xc) - xb + 0.5 * eps_b) / eps_b, 0.0, 1.0)
        s = u * u * u * (u * (6.0 * u - 15.0) + 10.0)
        Li = np.linalg.inv(np.linalg.cholesky((g * w) @ g.T))
        A = Li @ (0.5 * (dg * (w * (1.0 - s))) @ dg.T + (g * (w * (ven(x) + v_inf * s))) @ g.T) @ Li.T
        e, U = np.linalg.eigh(0.5 * (A + A.T))
        X = Li.T @ U[:, :M]
        X = X * np.where((g * (w * np.exp(0.37 * (x - xc)))).sum(1) @ X < 0, -1.0, 1.0)
        lam.append(e[:M])
        coef.append(X)
        gg, dd = table(cen, xg)
        F.append(X.T @ gg)
        dF.append(X.T @ dd)
    F, dF = np.concatenate(F), np.concatenate(dF)
    S1, h1, J1 = (F * wg) @ F.T, 0.5 * (dF * wg) @ dF.T + (F * (wg * ven(xg))) @ F.T, (F * (wg * xg)) @ F.T
    W = 1.0 / np.sqrt((xg[:, None] - xg) ** 2 + 0.25)
    pairs = np.zeros((L * L, K, 2), dtype=np.int32)
    for j in range(L):
        for i in range(L):
            cand = [(l, p) for l in range(M) for p in range(M) if i != j or l < p]
            e = [lam[i][l] + lam[j][p] for l, p in cand]
            tie = lambda u, v: abs(e[u] - e[v]) <= 1e-9 * (1.0 + abs(e[u]) + abs(e[v]))  # noqa: E731
            rank = [sum((cand[u] < cand[v]) if tie(u, v) else (e[u] < e[v]) for u in range(len(cand)) if u != v)
                    for v in range(len(cand))]
            pairs[i + L * j] = [cand[u] for u in np.argsort(rank)[:K]]
    S_, Hh, Gn = (np.zeros((L * L, K, K)) for _ in range(3))

    def gram(A, B, a0, b0, c0, d0):
        return A[np.ix_(a0, c0)] * B[np.ix_(b0, d0)]

    for o in range(L * L):
        i, j = o % L, o // L
        a0, b0 = i * M + pairs[o, :, 0], j * M + pairs[o, :, 1]
        S_[o] = gram(S1, S1, a0, b0, a0, b0) - gram(S1, S1, a0, b0, b0, a0)
        one = (gram(h1, S1, a0, b0, a0, b0) + gram(S1, h1, a0, b0, a0, b0) - gram(h1, S1, a0, b0, b0, a0)
               - gram(S1, h1, a0, b0, b0, a0))
        idx = sorted(set(range(i * M, i * M + M)) | set(range(j * M, j * M + M)))
        pos = {g: n for n, g in enumerate(idx)}
        n = len(idx)
        D = (F[idx][:, None, :] * F[idx][None, :, :]).reshape(n * n, -1) * wg
        E = (D @ W @ D.T).reshape(n, n, n, n)
        pa, pb = np.array([pos[v] for v in a0]), np.array([pos[v] for v in b0])
        Hh[o] = (one + E[pa[:, None], pa[None, :], pb[:, None], pb[None, :]]
                 - E[pa[:, None], pb[None, :], pb[:, None], pa[None, :]])
        if i + 1 < L:
            c0, d0 = (i + 1) * M + pairs[o + 1, :, 0], j * M + pairs[o + 1, :, 1]
            Gn[o] = gram(S1, S1, a0, b0, c0, d0) - gram(S1, S1, a0, b0, d0, c0)
    return {"lam": np.stack(lam), "coef": np.stack(coef), "S1": S1, "h1": h1, "J1": J1, "pairs": pairs, "S_lsd": S_,
            "H_lsd": Hh, "G_next": Gn}


def exact(case, seed):
    c, dev = dict(case), DEVICE if torch.cuda.is_available() else "cpu"
    kind = c["kind"]
    if kind in ("mlp_train", "mlp_predict"):
        return _exact_mlp(c, seed, kind == "mlp_train", dev)
    if kind == "lsd":
        return _exact_lsd(_lsd_args(c, seed))
    if kind == "traces":
        insts = P.learned_trace_family_16sd(c["instances"], seed)
        codes = [_exact_swr(i, c["kmax"], TOL, dev, (learn.CODE_S, learn.CODE_T))["codes"] for i in insts]
        return {"x": None, "codes": np.concatenate(codes), "done": None}
    if kind == "ground":
        r = _exact_swr(_instance(c, seed), c["kmax"], TOL, dev)
        return {"energy": np.array([r["energy"]]), "psi": r["psi"]}
    if kind == "time":
        r = _exact_swr(_instance(c, seed), 1, 0.0, dev)
        return {"res": r["res"][-1], "norm2": np.array([r["norm2"]]), "dipole": np.array([r["dipole"]]), "psi": r["psi"]}
    r = [_exact_swr(i, 1, 0.0, dev) for i in _batch(c, seed)]
    return {"res": np.array([v["res"][-1] for v in r]), "energy": np.array([v["energy"] for v in r]),
            "psi": np.concatenate([v["psi"] for v in r])}
