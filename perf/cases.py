"""Performance cases: calls that a user of the library makes, on device tensors.

Each case is a dict of plain values; `prepare` makes the load and the context
that a program keeps, `run` makes one call (or one short sequence of calls)
through the public binding, and `exact` states the same result in 64 bits with
torch alone. The loads are those of paper_2602_20787_gb300.ics: the
inverse-stereographic zoom-in load with its literal (wide) or 1:8 softening law,
optionally displaced or with a central filament, and the uniform ball of R^3.

Vectors come back whole, as (3, n) arrays. Accelerations and velocities of the
FP32 forms come back as float32: the entry points hand them over in float64
arrays, but they are computed in FP32, and a program that keeps them (a
snapshot, a tensor pipeline) stores that precision. Positions, and everything of
the FP64 form, stay float64.
"""
import math

import numpy as np
import torch

from paper_2602_20787_gb300 import ics, steps_cyl as sc

G = 1.0
L = 1.0
N0 = 4

_PRECISION = {"fp64": sc.STEPS_FP64, "kahan": sc.STEPS_FP32_KAHAN, "plain": sc.STEPS_FP32_PLAIN}


def _case(kind, n, **kw):
    """kind: force | kdk | noalloc | octree | r3 | train; tail: full | learned |
    table; law: literal (pair softenings up to several periods) | ratio8 (the
    production law, below 0.16 periods) | filament (a fifth of the particles in a
    dense line) | ball; a: scale factor (below 1: comoving masses and a^-3)."""
    c = {"kind": kind, "n": n, "n_cut": 64, "tail": "full", "precision": "kahan", "law": "literal", "a": 1.0,
         "steps": 0, "samples": 0, "epochs": 0}
    c.update(kw)
    return c


def listed():
    out = [
        # one force evaluation of the small static load: a convergence study or a
        # test problem, where latency and launches count as much as the pairs
        dict(_case("force", 2048), name="force_small"),
        # ten leapfrog steps of the same load from given positions, and the state back
        dict(_case("kdk", 2048, steps=10), name="kdk_small"),
        # the same load's FP64 reference force, against which the FP32 forms are judged
        dict(_case("force", 2048, precision="fp64"), name="force_fp64"),
        # the comoving run's force: displaced load at a = 0.02, 32 images, wide softening
        dict(_case("force", 65536, n_cut=16, a=0.02), name="force_lcdm"),
        # the large plain evaluation with all 128 images: the precision study's clustered load
        dict(_case("force", 200003, law="filament", a=0.02), name="force_filament"),
        # a production step as a driver program makes it: state in, one step with the
        # learned tail, state out (two force evaluations)
        dict(_case("kdk", 65536, law="ratio8", tail="learned", steps=1, a=1.0), name="kdk_learned"),
        # the correction-table tail on the wide softening law, odd size
        dict(_case("force", 80021, tail="table", a=0.02), name="force_table"),
        # the infinite window (no cut-off), an odd and middling size
        dict(_case("force", 30011, n_cut=0, tail="table", a=0.02), name="force_infinite"),
        # the tree code on the production load: build and walk
        dict(_case("octree", 262144, n_cut=0, tail="table", law="ratio8", a=0.02), name="force_octree"),
        # the isolated (R^3) topology
        dict(_case("r3", 65536, law="ball", n_cut=1), name="force_r3"),
        # pair accelerations for a program that may not allocate device memory
        dict(_case("noalloc", 10007, n_cut=16), name="pair_noalloc"),
        # training the learned tail: exact FP64 targets, forward, backward, Adam
        dict(_case("train", 16384, law="ratio8", a=0.02, samples=1 << 18, epochs=20), name="train_tail"),
    ]
    return out


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["force", "force", "force", "kdk", "tail", "tail", "inf", "octree", "r3", "noalloc", "fp64",
                       "train"])
    a = rng.choice([0.02, 0.1, 1.0])
    law = rng.choice(["literal", "ratio8", "filament"])
    n_cut = _log_int(rng, 8, 96)
    prec = rng.choice(["kahan", "kahan", "plain"])
    if kind == "force":
        return _case("force", _log_int(rng, 1000, 140000), n_cut=n_cut, law=law, a=a, precision=prec)
    if kind == "fp64":
        return _case("force", _log_int(rng, 600, 6000), n_cut=n_cut, law=law, a=a, precision="fp64")
    if kind == "kdk":
        n = _log_int(rng, 1000, 60000)
        return _case("kdk", n, n_cut=n_cut, law=law, precision=prec, steps=rng.randint(2, 10) if n < 12000 else 1)
    if kind == "tail":
        t = rng.choice(["learned", "table"])
        return _case("force", _log_int(rng, 4000, 120000), n_cut=_log_int(rng, 16, 96), law=law, a=a, tail=t,
                     precision=prec)
    if kind == "inf":
        return _case("force", _log_int(rng, 2000, 100000), n_cut=0, tail="table", law=law, a=a, precision=prec)
    if kind == "octree":
        return _case("octree", _log_int(rng, 20000, 400000), n_cut=0, tail="table", law="ratio8", a=a)
    if kind == "r3":
        return _case("r3", _log_int(rng, 2000, 200000), n_cut=1, law="ball", precision=prec)
    if kind == "noalloc":
        return _case("noalloc", _log_int(rng, 500, 60000), n_cut=n_cut, law=law, precision=prec)
    return _case("train", _log_int(rng, 4096, 30000), n_cut=_log_int(rng, 16, 96), law="ratio8", a=0.02,
                 samples=1 << rng.randint(17, 19), epochs=rng.randint(10, 20))


# ---- inputs ---------------------------------------------------------------------
def _load(case, seed):
    """The particle load (numpy, FP64) and its mean density."""
    n, law = case["n"], case["law"]
    if law == "ball":
        d = ics.ball_load(n, seed)
        return d, d["rho_bar"]
    comoving = case["a"] < 1.0
    rho = ics.comoving_rho_bar() if comoving else 1.0 / (math.pi * ics.R_SIM ** 2 * L)
    M = rho * math.pi * ics.R_SIM ** 2 * L
    d = ics.particle_load(n, seed, M, displaced=comoving or law != "literal", rho_bar=rho,
                          filament_frac=0.2 if law == "filament" else 0.0,
                          eps_law="ratio8" if law == "ratio8" else "literal")
    return d, rho


def _columns(d):
    dev = torch.device("cuda", torch.cuda.current_device())
    pos = torch.from_numpy(d["pos"]).to(dev)
    x, y, z = (pos[:, k].contiguous() for k in range(3))
    m, h = torch.from_numpy(d["m"]).to(dev), torch.from_numpy(d["h"]).to(dev)
    return x, y, z, m, h


_DT = 1e-3


class _State:
    """What a program keeps: the inputs, the outputs' arrays and the context."""

    def __init__(self):
        self.ctx = None

    def __del__(self):
        try:
            if self.ctx:
                sc.steps_cyl_free(self.ctx)
                self.ctx = None
        except Exception:
            pass


def prepare(case, seed):
    d, rho = _load(case, seed)
    n, kind = case["n"], case["kind"]
    s = _State()
    s.case = case
    s.cols = _columns(d)
    x, y, z, m, h = s.cols
    s.out = [torch.empty_like(x) for _ in range(6 if kind == "kdk" else 3)]
    s.stream = torch.cuda.current_stream().cuda_stream
    if kind == "noalloc":
        return s
    s.vel = [torch.zeros_like(x) for _ in range(3)]
    inf, r3 = case["n_cut"] == 0, kind == "r3"
    cfg = sc.Config(G=G, L=L, R_sim=2.0 if r3 else ics.R_SIM, rho_bar=rho, n_cut=case["n_cut"], n0=N0,
                    precision=_PRECISION[case["precision"]], tail=sc.STEPS_TAIL_TABLE if inf else sc.STEPS_TAIL_FULL,
                    background=sc.STEPS_BG_SPHERE if r3 else sc.STEPS_BG_INFINITE if inf else sc.STEPS_BG_FINITE,
                    comoving=case["a"] < 1.0, a_start=case["a"],
                    topology=sc.STEPS_TOPO_R3 if r3 else sc.STEPS_TOPO_S1R2,
                    force=sc.STEPS_FORCE_OCTREE if kind == "octree" else sc.STEPS_FORCE_DIRECT, stream=s.stream)
    s.ctx = sc.steps_cyl_init(cfg, n, x, y, z, *s.vel, m, h)
    if kind == "octree":
        # a program draws a new frame at each evaluation; here it is fixed, so that
        # a repeated pass builds the same tree
        sc.steps_cyl_tree_frame(s.ctx, 0.37, 1.1)
    if kind == "train":
        s.cfg = sc.steps_cyl_train_cfg_default(n_samples=case["samples"], epochs=case["epochs"], batch=4096,
                                               seed=seed & 0xffff, err_median=1e-4, err_p999=1e-2)
    elif case["tail"] == "learned":
        sc.steps_cyl_train_surrogate(s.ctx, sc.steps_cyl_train_cfg_default(n_samples=1 << 19, epochs=30))
        sc.steps_cyl_set_tail(s.ctx, sc.STEPS_TAIL_SURROGATE)
    elif case["tail"] == "table" and not inf:
        sc.steps_cyl_build_tail_table(s.ctx)
        sc.steps_cyl_set_tail(s.ctx, sc.STEPS_TAIL_TABLE)
    return s


def run(s):
    c, kind = s.case, s.case["kind"]
    if kind == "noalloc":
        sc.steps_cyl_pair_accel_noalloc(*s.cols, G, L, c["n_cut"], _PRECISION[c["precision"]], *s.out, stream=s.stream)
        return torch.stack(s.out).float()
    if kind == "train":
        sc.steps_cyl_train_surrogate(s.ctx, s.cfg)
        return sc.steps_cyl_get_surrogate(s.ctx)
    if kind == "kdk":
        sc.steps_cyl_set_state(s.ctx, *s.cols[:3], *s.vel)
        sc.steps_cyl_kdk_step(s.ctx, _DT, c["steps"])
        sc.steps_cyl_get_state(s.ctx, *s.out)
        return [torch.stack(s.out[:3]), torch.stack(s.out[3:]).float()]
    sc.steps_cyl_forces(s.ctx, *s.out)
    g = torch.stack(s.out)
    return g if c["precision"] == "fp64" else g.float()


# ---- floors ---------------------------------------------------------------------
def work(case):
    n, kind = case["n"], case["kind"]
    pairs = 0.5 * n * (n - 1.0)  # the force is symmetric: each unordered pair once
    b = 8.0 * n * (5 + 3)        # x, y, z, m, h in; three components out
    if kind == "r3":
        return {"bytes": b, "flops": 28.0 * pairs}
    if kind == "train":
        # 3 x forward flops per sample and epoch; the targets' FP64 image sums
        return {"bytes": 8.0 * n * 5 + 5 * 4.0 * case["samples"],
                "flops": case["samples"] * (case["epochs"] * 3 * 2368.0 + 2 * (case["n_cut"] - N0) * 12.0)}
    # an S1xR2 pair: the separation and both sides' sums (30), nine near images one
    # by one (9 each) and the rest of the image line, which has a closed form (80)
    per_pair = 30.0 + 9 * 9.0 + 80.0
    if kind == "octree":
        return {"bytes": b, "flops": per_pair * n * 110.0 * math.log2(n)}
    evals = case["steps"] + 1 if kind == "kdk" else 1
    if kind == "kdk":
        b = 8.0 * n * (8 + 6)
    return {"bytes": b, "flops": per_pair * pairs * evals}


# ---- the same results in 64 bits ---------------------------------------------------
def _spline_over_r(r2, hh):
    """F(r, h) / r of the softened force for h the support radius; 1 / r^3 outside."""
    r = torch.sqrt(r2)
    u = r / hh
    inner = (32.0 / 3.0 + u * u * (32.0 * u - 38.4)) / hh ** 3
    uo = torch.clamp(u, min=0.25)
    outer = (64.0 / 3.0 - 48.0 * uo + 38.4 * uo ** 2 - (32.0 / 3.0) * uo ** 3 - 1.0 / (15.0 * uo ** 3)) / hh ** 3
    return torch.where(u < 0.5, inner, torch.where(u < 1.0, outer, 1.0 / torch.clamp(r, min=1e-300) ** 3))


def _tail(x, R2):
    """Sums of (x + 1/2 + j, j = 0, 1, ...) images' 1/r^3 and z/r^3 from x on: the
    midpoint rule's Euler-Maclaurin series with three corrections."""
    i = 1.0 / torch.sqrt(x * x + R2)
    s = x * i
    q, e = s * s, i * i
    f1, f3, f5 = -3 * s * e * e, -15 * s * e ** 3 * (7 * q - 3), -315 * s * e ** 4 * ((33 * q - 30) * q + 5)
    i3 = e * i
    g1, g3 = -i3 * (3 * q - 1), -3 * i3 * e * ((35 * q - 30) * q + 3)
    g5 = -45 * i3 * e * e * (((231 * q - 315) * q + 105) * q - 5)
    return (e / (1 + s) + f1 / 24 - 7 * f3 / 5760 + 31 * f5 / 967680,
            i + g1 / 24 - 7 * g3 / 5760 + 31 * g5 / 967680)


def _window(dR2, dz, hh, n_cut, h_max):
    """sum F / r and sum z F / r over the window |dz + k| < n_cut (0: all images)."""
    near = 12 if n_cut == 0 or n_cut > 14 else n_cut
    near = max(near, int(math.ceil(h_max + 0.5)))
    near = min(near, n_cut) if n_cut else near
    direct = n_cut != 0 and near == n_cut
    sr, sz = torch.zeros_like(dz), torch.zeros_like(dz)
    for k in range(-near, near + 1):
        o = dz + k
        r2 = o * o + dR2
        if abs(k) - 0.5 <= h_max:
            f = _spline_over_r(r2, hh)
        else:
            ri = torch.rsqrt(r2)
            f = ri * ri * ri
        if direct and abs(k) == n_cut:
            f = f * (o.abs() < n_cut)
        sr += f
        sz += o * f
    if not direct:
        ua, za = _tail(near + 0.5 + dz, dR2)
        ub, zb = _tail(near + 0.5 - dz, dR2)
        sr += ua + ub
        sz += za - zb
        if n_cut:
            # the window ends at the images k with |dz + k| < n_cut: the largest is
            # n_cut - 1 above for dz >= 0 (n_cut for dz < 0) and mirrored below
            ha = torch.where(dz < 0, n_cut + 0.5, n_cut - 0.5) + dz
            hb = torch.where(dz > 0, n_cut + 0.5, n_cut - 0.5) - dz
            ua, za = _tail(ha, dR2)
            ub, zb = _tail(hb, dR2)
            sr -= ua + ub
            sz -= za - zb
    return sr, sz


def _pair_field(x, y, z, m, h, n_cut, r3):
    n = x.numel()
    acc = torch.empty(3, n, dtype=torch.float64, device=x.device)
    rows = max(1, (1 << 21) // n)
    h_max = float(2 * h.max())
    for a in range(0, n, rows):
        b = min(n, a + rows)
        dx, dy = x[a:b, None] - x, y[a:b, None] - y
        dz, hh = z[a:b, None] - z, h[a:b, None] + h
        dR2 = dx * dx + dy * dy
        if r3:
            sr = _spline_over_r(dR2 + dz * dz, hh)
            sz = dz * sr
        else:
            dz = dz - torch.round(dz / L) * L
            sr, sz = _window(dR2, dz, hh, n_cut, h_max)
        k = torch.arange(a, b, device=x.device)
        sr[k - a, k] = 0.0
        sz[k - a, k] = 0.0
        acc[0, a:b] = -G * ((dx * sr) @ m)
        acc[1, a:b] = -G * ((dy * sr) @ m)
        acc[2, a:b] = -G * (sz @ m)
    return acc


def _background(x, y, rho0, n_cut):
    """-F_h(rho) rho_hat of the homogeneous cylinder of radius R and half height
    n_cut L (0: infinite), by Gauss-Legendre quadrature of its finite-height part."""
    R = ics.R_SIM
    rho = torch.sqrt(x * x + y * y)
    F = torch.where(rho <= R, -2 * math.pi * G * rho0 * rho, -2 * math.pi * G * rho0 * R * R / rho)
    if n_cut:
        t, w = np.polynomial.legendre.leggauss(400)
        t, w = 0.25 * math.pi * (t + 1), 0.25 * math.pi * w
        Lw = n_cut * L
        for th, wt in zip(t, w):
            q = 4 * rho * R * math.sin(0.5 * th) ** 2
            A, B = (R + rho) ** 2 - q, (R - rho) ** 2 + q
            lg = torch.log((torch.sqrt(Lw * Lw + A) + Lw) / (torch.sqrt(Lw * Lw + B) + Lw))
            F = F + 4 * G * rho0 * wt * R * math.cos(th) * lg
    return -F * x / rho, -F * y / rho


def exact(case, seed):
    n, kind = case["n"], case["kind"]
    evals = case["steps"] + 1 if kind == "kdk" else 1
    if kind in ("octree", "train") or float(n) * n * evals > (4e10 if kind == "r3" else 9e9):
        return None
    d, rho0 = _load(case, seed)
    x, y, z, m, h = _columns(d)

    def field(x, y, z):
        g = _pair_field(x, y, z, m, h, case["n_cut"], kind == "r3")
        if kind == "r3":
            c = 4.0 * math.pi * G * rho0 / 3.0
            g += c * torch.stack([x, y, z])
        elif kind != "noalloc":
            bx, by = _background(x, y, rho0, case["n_cut"])
            g[0] += bx
            g[1] += by
        return g / case["a"] ** 3

    if kind != "kdk":
        return field(x, y, z)
    v = torch.zeros(3, n, dtype=torch.float64, device=x.device)
    g = field(x, y, z)
    for _ in range(case["steps"]):
        v += 0.5 * _DT * g
        x, y, z = x + _DT * v[0], y + _DT * v[1], torch.remainder(z + _DT * v[2], L)
        g = field(x, y, z)
        v += 0.5 * _DT * g
    return [torch.stack([x, y, z]), v]
