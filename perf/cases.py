"""The work a user of this library has it do, as cases to be timed.

Whole fits (one small subject, the 1 mm volume, a batch of small subjects)
and the calls a program that runs its own updates makes: the voxel pass, the
JTV reweighting, the Newton-system solve with either preconditioner, the
Laplace uncertainty and the voxel pass of scans that moved.  Sizes are those
of the benchmark (64^3, 1 mm 176 x 240 x 256, 0.8 mm 208 x 300 x 320) and of
the tests, and a 1 mm head cropped to odd dimensions (181 x 217 x 181).

Inputs follow the library's synthetic recipe (Voronoi regions with a smooth
modulation, B1 fields, Rician noise at first-echo SNR 20), drawn on the GPU
from the seed.  Everything that feeds a case, and `exact`, is plain torch.
"""
import math
import random

import numpy as np
import torch

import paper_2102_01604_gb300 as mpm

# nominal flip angle (degrees), TR (s), MT pulse
CONTRASTS = {"PDw": (6.0, 0.025, 0), "T1w": (21.0, 0.025, 0), "MTw": (6.0, 0.025, 1),
             "VFA15": (15.0, 0.025, 0)}
ECHO_SPACING = 0.0023                # s
SNR = 20.0
LAMBDA, EPS = 10.0, 1e-3
MPM3 = {"contrasts": "PDw,T1w,MTw", "echoes": "8,8,6"}      # the paper's protocol
VFA2 = {"contrasts": "PDw,T1w", "echoes": "6,6"}            # two flip angles, no MT: three maps


def listed():
    mm1 = {"nx": 176, "ny": 240, "nz": 256, "vx": 1.0, **MPM3}
    return [
        # one small subject, start to finish: a chain of some 700 short kernels
        {"name": "fit 64^3", "kind": "fit", "nx": 64, "ny": 64, "nz": 64, "vx": 1.0, **MPM3,
         "gn": 20, "cg": 30},
        # one 1 mm subject, start to finish: what most users run
        {"name": "fit 1 mm", "kind": "fit", **mm1, "gn": 20, "cg": 30},
        # a queue of small subjects fitted together
        {"name": "batch 16 x 64^3", "kind": "batch", "shapes": ",".join(["64x64x64"] * 16), "vx": 1.0,
         **MPM3, "gn": 20, "cg": 30},
        # one Newton system of the 1 mm volume: nearly all the time of a fit
        {"name": "solve 1 mm", "kind": "solve", **mm1, "cg": 30},
        # the same system on a head cropped to odd dimensions
        {"name": "solve odd 181x217x181", "kind": "solve", "nx": 181, "ny": 217, "nz": 181, "vx": 1.0,
         **MPM3, "cg": 30},
        # a small region of interest, no MT contrast (three maps): latency and launches
        {"name": "solve small 48x40x20", "kind": "solve", "nx": 48, "ny": 40, "nz": 20, "vx": 1.0, **VFA2,
         "cg": 30},
        # an early update solved to about 1e-3 with the multigrid preconditioner
        {"name": "solve multigrid 1 mm", "kind": "mg", **mm1, "cg": 12},
        # gradient, Hessian and likelihood of the 1 mm images
        {"name": "voxel pass 1 mm", "kind": "grad_hess", **mm1, "dtype": "f32", "precond": 0},
        # the same of 0.8 mm images kept in bfloat16
        {"name": "voxel pass 0.8 mm bf16", "kind": "grad_hess", "nx": 208, "ny": 300, "nz": 320, "vx": 0.8,
         **MPM3, "dtype": "bf16", "precond": 0},
        # the prior's weights and energy
        {"name": "jtv 1 mm", "kind": "jtv", **mm1},
        # error bars: variances, log-determinant and moments at the final maps
        {"name": "uncertainty 1 mm", "kind": "uncertainty", **mm1},
        # the voxel pass of contrasts that moved between the scans
        {"name": "moved voxel pass 1 mm", "kind": "moved", **mm1, "dtype": "f32", "precond": 0},
    ]


def _dims(rng, lo, hi):
    """Dimensions of a volume of lo..hi voxels (uniform in the logarithm);
    half have an x size that is a multiple of 4, as scanner matrices have, the
    others are cropped anywhere."""
    n = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    f = [math.exp(rng.uniform(-0.25, 0.25)) for _ in range(3)]
    s = (n / (f[0] * f[1] * f[2])) ** (1 / 3)
    d = [max(8, round(s * v)) for v in f]
    if rng.random() < 0.5:
        d[0] = max(8, 4 * round(d[0] / 4))
    return {"nx": d[0], "ny": d[1], "nz": d[2], "vx": rng.choice([0.8, 1.0])}


def draw(rng):
    kind = rng.choice(["fit", "batch", "solve", "solve", "mg", "grad_hess", "grad_hess", "jtv",
                       "uncertainty", "moved"])
    prot = rng.choice([MPM3, MPM3, VFA2, {"contrasts": "PDw,T1w,MTw,VFA15", "echoes": "6,6,5,4"}])
    if kind == "batch":
        ds = [_dims(rng, 3e4, 4e5) for _ in range(rng.randint(2, 8))]
        return {"kind": kind, "shapes": ",".join("%dx%dx%d" % (d["nx"], d["ny"], d["nz"]) for d in ds),
                "vx": 1.0, **prot, "gn": rng.randint(5, 15), "cg": rng.choice([20, 30])}
    if kind == "fit":
        return {"kind": kind, **_dims(rng, 2e4, 1.5e6), **prot, "gn": rng.randint(5, 20),
                "cg": rng.choice([10, 20, 30])}
    if kind == "solve":
        return {"kind": kind, **_dims(rng, 2e4, 2e7), **prot, "cg": rng.randint(10, 32)}
    if kind == "mg":
        return {"kind": kind, **_dims(rng, 1e5, 1e7), **prot, "cg": rng.randint(4, 12)}
    c = {"kind": kind, **_dims(rng, 2e4, 1e7 if kind == "moved" else 2e7), **prot}
    if kind in ("grad_hess", "moved"):
        c.update(dtype=rng.choice(["f32", "bf16"]), precond=rng.choice([0, 0, 1]))
    return c


# ------------------------------------------------------------------ inputs

def _f32(v):
    return float(np.float32(v))


def _protocol(case):
    """Flip angle, TR, MT, echo counts and times, rounded to the float32 the
    library computes in."""
    names = case["contrasts"].split(",")
    ne = [int(v) for v in case["echoes"].split(",")]
    return {"alpha": [_f32(math.radians(CONTRASTS[c][0])) for c in names],
            "tr": [_f32(CONTRASTS[c][1]) for c in names], "mt": [CONTRASTS[c][2] for c in names],
            "n_echoes": ne, "te": [_f32(ECHO_SPACING * (k + 1)) for n in ne for k in range(n)],
            "sigma2": [1.0] * len(names)}


def _outer(fx, fy, fz):
    return (fz[:, None, None] * fy[None, :, None] * fx[None, None, :]).reshape(-1)


def _field(rng, shape, dev):
    """A product of low-frequency cosines, scaled to [-1, 1], flat with x fastest."""
    f = []
    for n in shape:
        a = torch.arange(n, device=dev, dtype=torch.float32) / n
        c = torch.cos(math.pi * rng.randint(1, 2) * a + rng.uniform(0, 2 * math.pi))
        f.append(c / c.abs().max().clamp_min(1e-6))
    return _outer(*f)


def _truth(rng, shape, K, dev):
    """Log-parameter maps [K, N]: 12 Voronoi regions, each map modulated by 5%."""
    ax = [torch.arange(n, device=dev, dtype=torch.float32) / n for n in shape]
    best = torch.full((shape[2], shape[1], shape[0]), float("inf"), device=dev)
    label = torch.zeros_like(best, dtype=torch.int64)
    for r in range(12):
        c = [rng.random() for _ in range(3)]
        d = (((ax[2] - c[2]) ** 2)[:, None, None] + ((ax[1] - c[1]) ** 2)[None, :, None]
             + ((ax[0] - c[0]) ** 2)[None, None, :])
        label[d < best] = r
        best = torch.minimum(best, d)
    label = label.reshape(-1)
    y = []
    for lo, hi in [(2000.0, 4000.0), (0.5, 1.5), (10.0, 40.0), (0.002, 0.02)][:K]:
        v = torch.tensor([rng.uniform(lo, hi) for _ in range(12)], device=dev)[label]
        v = v * (1.0 + 0.05 * _field(rng, shape, dev))
        y.append(torch.log(v / (1.0 - v)) if len(y) == 3 else torch.log(v))
    return torch.stack(y)


def _terms(prot, c, y, bp):
    """The factors of contrast c shared by its echoes (signal at TE = 0 without
    B1-, and the derivatives' factors), in the type of y."""
    a, r1 = torch.exp(y[0]), torch.exp(y[1])
    d = torch.sigmoid(y[3]) if prot["mt"][c] else torch.zeros_like(a)
    m = torch.sigmoid(-y[3]) if prot["mt"][c] else torch.ones_like(a)
    ang = prot["alpha"][c] * bp
    sa, ca = torch.sin(ang), torch.cos(ang)
    tt = prot["tr"][c] * r1
    E, omE = torch.exp(-tt), -torch.expm1(-tt)
    D = 1 - m * ca * E
    return {"s0": a * sa * m * omE / D, "q1": tt * E * (1 - m * ca) / (omE * D), "qd": -d / D,
            "h1": 1 - tt * (2 - D) / D, "hd": 2 * m * (1 - ca * E) / D - 1,
            "cross": tt * E * ca * d * m / (D * D)}


def _scan(prot, c, y, bp, bm, gen):
    """Noisy echoes [E, N] (float32) of contrast c; fills in its noise variance."""
    i0, ne = sum(prot["n_echoes"][:c]), prot["n_echoes"][c]
    s0 = _terms(prot, c, y, bp)["s0"] * bm
    r2 = torch.exp(y[2])
    first = s0 * torch.exp(-prot["te"][i0] * r2)
    sig = float(first.mean()) / SNR
    prot["sigma2"][c] = _f32(sig * sig)
    x = torch.empty((ne, y.shape[1]), device=y.device)
    for e in range(ne):
        s = s0 * torch.exp(-prot["te"][i0 + e] * r2)
        n1 = torch.randn(s.shape, generator=gen, device=s.device)
        n2 = torch.randn(s.shape, generator=gen, device=s.device)
        x[e] = torch.sqrt((s + sig * n1) ** 2 + (sig * n2) ** 2)
    return x


def _subject(case, shape, seed, noise=0.01):
    """Images, B1 fields and maps of one subject; `y` are maps part way through
    a fit (the truth with a little noise)."""
    dev = torch.device("cuda")
    rng = random.Random(seed)
    gen = torch.Generator(device=dev)
    gen.manual_seed(seed)
    prot = _protocol(case)
    K = 4 if any(prot["mt"]) else 3
    truth = _truth(rng, shape, K, dev)
    N = truth.shape[1]
    C = len(prot["alpha"])
    bp = 1.0 + 0.2 * _field(rng, shape, dev)
    bm = torch.stack([1.0 + 0.1 * _field(rng, shape, dev) for _ in range(C)])
    x = torch.cat([_scan(prot, c, truth, bp, bm[c], gen) for c in range(C)])
    if case.get("dtype") == "bf16":
        x = x.to(torch.bfloat16)
    y = truth + noise * torch.randn((K, N), generator=gen, device=dev)
    return {"prot": prot, "shape": shape, "K": K, "N": N, "x": x, "b1p": bp.contiguous(), "b1m": bm, "y": y}


def _shape(case):
    return case["nx"], case["ny"], case["nz"]


# the scans' motion: rotations (degrees, axis) and shifts (voxels) of the 2nd,
# 3rd and 4th contrast against the first
MOTION = [(0.0, 2, (0.0, 0.0, 0.0)), (2.0, 2, (1.5, -1.0, 0.5)), (3.0, 0, (-0.75, 2.0, 1.0)),
          (-1.5, 1, (0.5, 0.25, -1.0))]


def _affines(shape, C):
    """Per contrast the 3 x 4 map from its voxels to reconstruction voxels: a
    rotation about the centre, then a shift (float32 values)."""
    ctr = (np.array(shape, dtype=np.float64) - 1) / 2
    out = []
    for deg, axis, shift in MOTION[:C]:
        t = math.radians(deg)
        R = np.eye(3)
        i, j = [k for k in range(3) if k != axis]
        R[i, i] = R[j, j] = math.cos(t)
        R[i, j], R[j, i] = -math.sin(t), math.sin(t)
        A = np.concatenate([R, (ctr - R @ ctr + np.array(shift))[:, None]], axis=1)
        out.append(A.astype(np.float32).astype(np.float64))
    return out


def _cells(shape, A, dtype):
    """Cell corners, offsets and the inside mask of every acquisition voxel."""
    nx, ny, nz = shape
    dev = torch.device("cuda")
    k, j, i = torch.meshgrid(*[torch.arange(n, device=dev, dtype=dtype) for n in (nz, ny, nx)], indexing="ij")
    r = [(A[d, 0] * i + A[d, 1] * j + A[d, 2] * k + A[d, 3]).reshape(-1) for d in range(3)]
    inside = torch.ones_like(r[0], dtype=torch.bool)
    for d in range(3):
        inside &= (r[d] >= 0) & (r[d] <= shape[d] - 1)
    b = [torch.floor(v) for v in r]
    return [v.long() for v in b], [v - w for v, w in zip(r, b)], inside


def _corners(shape, b, f, inside):
    """(weight, voxel index) of the 8 corners of every cell; 0 outside."""
    nx, ny, nz = shape
    for cz in (0, 1):
        for cy in (0, 1):
            for cx in (0, 1):
                w = (f[0] if cx else 1 - f[0]) * (f[1] if cy else 1 - f[1]) * (f[2] if cz else 1 - f[2])
                X, Y, Z = b[0] + cx, b[1] + cy, b[2] + cz
                ok = inside & (X < nx) & (Y < ny) & (Z < nz)
                yield torch.where(ok, w, torch.zeros_like(w)), torch.where(ok, X + nx * (Y + ny * Z), 0)


def _pull(shape, A, u):
    b, f, inside = _cells(shape, A, u.dtype)
    out = torch.zeros_like(u)
    for w, n in _corners(shape, b, f, inside):
        for k in range(u.shape[0]):
            out[k] += w * u[k][n]
    return out, inside


def _moved(case, seed):
    """Scans that moved: contrast c sees the maps through its own affine."""
    dev = torch.device("cuda")
    shape = _shape(case)
    rng = random.Random(seed)
    gen = torch.Generator(device=dev)
    gen.manual_seed(seed)
    prot = _protocol(case)
    K = 4 if any(prot["mt"]) else 3
    truth = _truth(rng, shape, K, dev)
    affs = _affines(shape, len(prot["alpha"]))
    xs, bps, bms = [], [], []
    for c, A in enumerate(affs):
        yc, inside = _pull(shape, A, truth)
        yc = torch.where(inside[None], yc, truth.mean(dim=1, keepdim=True))
        bps.append((1.0 + 0.2 * _field(rng, shape, dev)).contiguous())
        bms.append((1.0 + 0.1 * _field(rng, shape, dev)).contiguous())
        x = _scan(prot, c, yc, bps[c], bms[c], gen)
        xs.append(x.to(torch.bfloat16) if case["dtype"] == "bf16" else x)
    y = truth + 0.01 * torch.randn(truth.shape, generator=gen, device=dev)
    return {"prot": prot, "shape": shape, "K": K, "N": truth.shape[1], "xs": xs, "b1ps": bps, "b1ms": bms,
            "affines": affs, "y": y}


def _problem(case, d):
    return mpm.make_problem(d["prot"], d["shape"], vx=[case["vx"]] * 3, lam=LAMBDA, eps=EPS,
                            precond=case.get("precond", 0),
                            echo_dtype=1 if case.get("dtype") == "bf16" else 0)


# a tolerance-limited multigrid solve as the benchmark runs it
MG = dict(mg_levels=8, mg_nu=1, mg_omega=0.7, mg_coarse_sweeps=20)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        subs = []
        for i, t in enumerate(case["shapes"].split(",")):
            d = _subject(case, tuple(int(v) for v in t.split("x")), 1000 * seed + i)
            subs.append((d, _problem(case, d)))
        opts = mpm.make_opts(gn_iters=case["gn"], cg_iters=case["cg"], graph="phased")
        return {"kind": kind, "opts": opts, "problems": [p for _, p in subs],
                "xs": [d["x"] for d, _ in subs], "b1ps": [d["b1p"] for d, _ in subs],
                "b1ms": [d["b1m"] for d, _ in subs], "ys": [torch.zeros_like(d["y"]) for d, _ in subs],
                "vars": [torch.empty_like(d["y"]) for d, _ in subs],
                "wss": [mpm.workspace(p, opts) for _, p in subs]}
    if kind == "moved":
        d = _moved(case, seed)
        p = _problem(case, d)
        proj = mpm.make_projection([d["shape"]] * len(d["xs"]), d["affines"])
        return {"kind": kind, "p": p, "proj": proj, "ws": mpm.workspace_proj(p, proj, None, mpm._lib.CALL_GRAD_HESS),
                **{k: d[k] for k in ("xs", "b1ps", "b1ms", "y")}}
    d = _subject(case, _shape(case), seed)
    p = _problem(case, d)
    s = {"kind": kind, "p": p}
    if kind == "fit":
        opts = mpm.make_opts(gn_iters=case["gn"], cg_iters=case["cg"])
        s.update(opts=opts, x=d["x"], b1p=d["b1p"], b1m=d["b1m"], y=torch.zeros_like(d["y"]),
                 var=torch.empty_like(d["y"]), ws=mpm.workspace(p, opts))
    elif kind in ("solve", "mg"):
        g, h, _ = _grad_hess64(d, case.get("precond", 0))
        opts = mpm.make_opts(cg_iters=case["cg"], **(MG if kind == "mg" else {}))
        s.update(opts=opts, g=g.float(), h=h.float(), w=_jtv64(d, case["vx"])[0].float(), y=d["y"],
                 delta=torch.empty_like(d["y"]),
                 resid=torch.full((case["cg"] + 1,), float("nan"), dtype=torch.float64, device="cuda"),
                 ws=mpm.workspace(p, opts, mpm._lib.CALL_SOLVE))
    elif kind == "grad_hess":
        T = d["K"] * (d["K"] + 1) // 2
        s.update(x=d["x"], y=d["y"], b1p=d["b1p"], b1m=d["b1m"], g=torch.empty_like(d["y"]),
                 h=torch.empty((T, d["N"]), device="cuda"),
                 nll=torch.empty(1, dtype=torch.float64, device="cuda"),
                 ws=mpm.workspace(p, None, mpm._lib.CALL_GRAD_HESS))
    elif kind == "jtv":
        s.update(y=d["y"], w=torch.empty(d["N"], device="cuda"),
                 jtv=torch.empty(1, dtype=torch.float64, device="cuda"),
                 ws=mpm.workspace(p, None, mpm._lib.CALL_JTV))
    else:
        _, h, _ = _grad_hess64(d, 0)
        s.update(h=h.float(), w=_jtv64(d, case["vx"])[0].float(), y=d["y"], var=torch.empty_like(d["y"]),
                 logdet=torch.empty(d["N"], device="cuda"), moments=torch.empty((4, d["N"]), device="cuda"))
    return s


def run(s):
    kind = s["kind"]
    if kind == "fit":
        _, rep = mpm.mpm_fit(s["p"], s["opts"], s["x"], s["y"], s["b1p"], s["b1m"], var=s["var"], ws=s["ws"])
        return {"y": s["y"], "var": s["var"], "F": list(rep.F[:rep.iters + 1])}
    if kind == "batch":
        _, reps = mpm.mpm_fit_batch(s["problems"], s["opts"], s["xs"], s["ys"], s["b1ps"], s["b1ms"],
                                    s["vars"], s["wss"])
        return {"y": s["ys"], "var": s["vars"], "F": [r.F[r.iters] for r in reps]}
    if kind in ("solve", "mg"):
        delta, resid = mpm.mpm_solve(s["p"], s["opts"], s["h"], s["w"], s["g"], s["y"], delta=s["delta"],
                                     resid=s["resid"], ws=s["ws"])
        # a log of the convergence, kept at the precision the solve works in
        return {"delta": delta, "resid": resid.float()}
    if kind == "grad_hess":
        g, h, nll = mpm.mpm_grad_hess(s["p"], s["x"], s["y"], s["b1p"], s["b1m"], g=s["g"], h=s["h"],
                                      nll=s["nll"], ws=s["ws"])
        return {"g": g, "h": h, "nll": nll}
    if kind == "jtv":
        w, jtv = mpm.mpm_jtv_weights(s["p"], s["y"], w=s["w"], jtv=s["jtv"], ws=s["ws"])
        return {"w": w, "jtv": jtv}
    if kind == "uncertainty":
        var, logdet, moments = mpm.mpm_uncertainty(s["p"], s["h"], s["w"], s["y"], var=s["var"],
                                                   logdet=s["logdet"], moments=s["moments"],
                                                   want_moments=True)
        return {"var": var, "logdet": logdet, "moments": moments}
    g, h, nll = mpm.mpm_grad_hess_proj(s["p"], s["proj"], s["xs"], s["y"], s["b1ps"], s["b1ms"], ws=s["ws"])
    return {"g": g, "h": h, "nll": nll}


# ------------------------------------------------------------------ work

def work(case):
    """Bytes and flops of one pass: every input read once and every output
    written once; an iterative solve needs, in every iteration, its matrix
    (H and the weights) once and the state of conjugate gradient (solution,
    residual and direction) read and written once."""
    prot = _protocol(case)
    K = 4 if any(prot["mt"]) else 3
    T, I, C = K * (K + 1) // 2, sum(prot["n_echoes"]), len(prot["alpha"])
    eb = 2 if case.get("dtype") == "bf16" else 4
    shapes = ([tuple(int(v) for v in t.split("x")) for t in case["shapes"].split(",")]
              if case["kind"] == "batch" else [_shape(case)])
    N = sum(a * b * c for a, b, c in shapes)
    vox = (I * eb + 4 * (K + 1 + C) + 4 * (K + T), 20 * I + 60 * C + 6 * T)    # voxel pass, per voxel
    jtv = (4 * (K + 1), 24 * K)
    it = (4 * (T + 1) + 6 * 4 * K, 2 * K * K * 3 + 22 * K + 2 * T)             # one CG iteration
    ends = (4 * (T + 1 + 3 * K), 22 * K + 2 * K * K)                           # right-hand side, result
    unc = (4 * (T + 1 + K), 6 * T * K)
    kind = case["kind"]
    if kind in ("fit", "batch"):
        gn, cg = case["gn"], case["cg"]
        per = [(gn + 1) * (vox[i] + jtv[i]) + gn * (cg * it[i] + ends[i]) + unc[i] for i in (0, 1)]
    elif kind == "solve":
        per = [case["cg"] * it[i] + ends[i] for i in (0, 1)]
    elif kind == "mg":
        # per iteration the matrix is applied in the cycle before and after the
        # coarse correction too, to one vector read and written; coarse levels add a seventh
        cyc = (2 * (4 * (T + 1) + 2 * 4 * K), 2 * (2 * K * K * 2 + 22 * K))
        per = [case["cg"] * (it[i] + cyc[i] * 8 / 7) + ends[i] for i in (0, 1)]
    elif kind == "jtv":
        per = jtv
    elif kind == "uncertainty":
        per = (unc[0] + 4 * (1 + 4 + 1), unc[1] + 20)
    elif kind == "moved":
        # each scan has its own B1+; every scan's gradient and Hessian terms are spread over 8 voxels
        per = (vox[0] + 4 * (C - 1), vox[1] + C * 16 * (2 * K + T))
    else:
        per = vox
    return {"bytes": N * per[0], "flops": N * per[1]}


# ------------------------------------------------------------------ in 64 bits

def _contrast64(prot, c, K, x, y, bp, bm, precond):
    """Gradient [K, N], loaded Hessian [T, N] and likelihood of contrast c."""
    t = _terms(prot, c, y, bp)
    i0, ne = sum(prot["n_echoes"][:c]), prot["n_echoes"][c]
    is2 = 1.0 / prot["sigma2"][c]
    r2 = torch.exp(y[2])
    s0 = t["s0"] * bm
    z = torch.zeros_like(r2)
    S0, S1, S2, R0, R1, N2, A0, A2, B1 = (z.clone() for _ in range(9))
    for e in range(ne):
        q2 = -prot["te"][i0 + e] * r2
        s = s0 * torch.exp(q2)
        r = s - x[e].double()
        a = (r * s).abs()
        S0 += s * s
        S1 += s * s * q2
        S2 += (s * q2) ** 2
        R0 += r * s
        R1 += r * s * q2
        N2 += r * r
        A0 += a
        A2 += a * ((1 + q2) * q2).abs()
        B1 += a * q2.abs()
    q = [None, t["q1"], None, t["qd"]]
    g = [R0, R0 * q[1], R1, R0 * q[3]][:K]
    H = {(0, 0): S0, (0, 1): S0 * q[1], (0, 2): S1, (1, 1): S0 * q[1] ** 2, (1, 2): S1 * q[1], (2, 2): S2}
    if K == 4:
        H.update({(0, 3): S0 * q[3], (1, 3): S0 * q[1] * q[3], (2, 3): S1 * q[3], (3, 3): S0 * q[3] ** 2})
    a1, ad = q[1].abs(), q[3].abs()
    h1, hd = (t["h1"] * q[1]).abs(), (t["hd"] * q[3]).abs()
    load = [A0, A0 * h1, A2, A0 * hd]
    if precond == 1:
        c13 = (q[1] * q[3] + t["cross"]).abs()
        load = [A0 * (1 + a1 + ad) + B1, A0 * (h1 + a1 + c13) + a1 * B1, A2 + B1 * (1 + a1 + ad),
                A0 * (hd + ad + c13) + ad * B1]
    h = []
    for i in range(K):
        for j in range(i, K):
            h.append(H[(i, j)] + load[i] if i == j else H[(i, j)])
    return is2 * torch.stack(g), is2 * torch.stack(h), 0.5 * is2 * N2.sum()


def _grad_hess64(d, precond, y=None):
    prot, K = d["prot"], d["K"]
    y = d["y"].double() if y is None else y
    bp = d["b1p"].double()
    g = h = nll = 0.0
    for c in range(len(prot["alpha"])):
        i0 = sum(prot["n_echoes"][:c])
        gc, hc, nc = _contrast64(prot, c, K, d["x"][i0:i0 + prot["n_echoes"][c]], y, bp,
                                 d["b1m"][c].double(), precond)
        g, h, nll = g + gc, h + hc, nll + nc
    return g, h, nll.reshape(1)


def _vol(shape, v):
    return v.reshape(*v.shape[:-1], shape[2], shape[1], shape[0])


def _sides(v, ax):
    """The lower and upper ends of every edge along axis ax (-1: x, -2: y, -3: z)."""
    n = v.shape[ax]
    return v.narrow(ax, 0, n - 1), v.narrow(ax, 1, n - 1)


def _jtv64(d, vx, y=None):
    y = _vol(d["shape"], d["y"].double() if y is None else y)
    u = torch.zeros_like(y[0])
    for ax in (-1, -2, -3):
        lo, hi = _sides(y, ax)
        e = LAMBDA * ((hi - lo) ** 2).sum(0) / vx ** 2
        a, b = _sides(u, ax)
        a += e
        b += e
    s = torch.sqrt(u + _f32(EPS * EPS))
    return (1 / s).reshape(-1), s.sum().reshape(1)


class _System:
    """(H + L) of one level with its block preconditioner, in 64 bits.  Fields
    are [K, nz, ny, nx]; kap holds the edge coefficients along x, y and z."""

    def __init__(self, h, kap):
        self.h, self.kap, self.K = h, kap, {6: 3, 10: 4}[h.shape[0]]
        dsum = torch.zeros_like(h[0])
        for ax, k in zip((-1, -2, -3), kap):
            a, b = _sides(dsum, ax)
            a += k
            b += k
        self.dsum = dsum
        K = self.K
        M = self.block = [[None] * K for _ in range(K)]
        t = 0
        for i in range(K):
            for j in range(i, K):
                M[i][j] = M[j][i] = h[t] + (LAMBDA * dsum if i == j else 0.0)
                t += 1
        L = self.L = [[None] * K for _ in range(K)]
        for j in range(K):
            L[j][j] = torch.sqrt(M[j][j] - sum(L[j][k] ** 2 for k in range(j)))
            for i in range(j + 1, K):
                L[i][j] = (M[i][j] - sum(L[i][k] * L[j][k] for k in range(j))) / L[j][j]

    def edges(self, v):
        out = torch.zeros_like(v)
        for ax, k in zip((-1, -2, -3), self.kap):
            lo, hi = _sides(v, ax)
            f = k * (lo - hi)
            a, b = _sides(out, ax)
            a += f
            b -= f
        return LAMBDA * out

    def apply(self, v):
        out = self.edges(v)
        t = 0
        for i in range(self.K):
            for j in range(i, self.K):
                out[i] += self.h[t] * v[j]
                if i != j:
                    out[j] += self.h[t] * v[i]
                t += 1
        return out

    def precond(self, r):
        K, L = self.K, self.L
        t = []
        for i in range(K):
            t.append((r[i] - sum(L[i][k] * t[k] for k in range(i))) / L[i][i])
        z = [None] * K
        for i in reversed(range(K)):
            z[i] = (t[i] - sum(L[k][i] * z[k] for k in range(i + 1, K))) / L[i][i]
        return torch.stack(z)


def _system(shape, vx, h, w):
    wv = _vol(shape, w)
    kap = [sum(_sides(wv, ax)) / vx ** 2 for ax in (-1, -2, -3)]
    return _System(_vol(shape, h), kap)


def _pool(v):
    """Sums over 2 x 2 x 2 voxels (fewer at the far faces)."""
    for ax in (-1, -2, -3):
        n = v.shape[ax]
        if n % 2:
            v = torch.cat([v, torch.zeros_like(v.narrow(ax, 0, 1))], dim=ax)
        v = v.unflatten(ax, (v.shape[ax] // 2, 2)).sum(ax)
    return v


def _coarsen(S):
    kap = []
    for i, ax in enumerate((-1, -2, -3)):
        k = S.kap[i]
        n = k.shape[ax]
        # the edges that cross between coarse voxels, summed over the other two axes
        k = k.index_select(ax, torch.arange(1, n, 2, device=k.device))
        for other in (-1, -2, -3):
            if other != ax:
                m = k.shape[other]
                if m % 2:
                    k = torch.cat([k, torch.zeros_like(k.narrow(other, 0, 1))], dim=other)
                k = k.unflatten(other, (k.shape[other] // 2, 2)).sum(other)
        kap.append(k)
    return _System(_pool(S.h), kap)


def _vcycle(levels, l, r):
    S, om = levels[l], MG["mg_omega"]
    x = om * S.precond(r)
    if l == len(levels) - 1:
        for _ in range(MG["mg_coarse_sweeps"] - 1):
            x = x + om * S.precond(r - S.apply(x))
        return x
    for _ in range(MG["mg_nu"] - 1):
        x = x + om * S.precond(r - S.apply(x))
    e = _vcycle(levels, l + 1, _pool(r - S.apply(x)))
    for ax in (-1, -2, -3):
        e = e.repeat_interleave(2, dim=ax).narrow(ax, 0, x.shape[ax])
    x = x + e
    for _ in range(MG["mg_nu"]):
        x = x + om * S.precond(r - S.apply(x))
    return x


def _cg64(shape, vx, h, w, g, y, iters, multigrid=False):
    """delta [K, N] and the residual norms of preconditioned CG from zero."""
    S = _system(shape, vx, h, w)
    prec = S.precond
    if multigrid:
        levels = [S]
        while len(levels) < MG["mg_levels"] and levels[-1].h[0].numel() > 512:
            levels.append(_coarsen(levels[-1]))
        prec = lambda r: _vcycle(levels, 0, r)  # noqa: E731
    r = _vol(shape, g) + S.edges(_vol(shape, y))
    x = torch.zeros_like(r)
    z = prec(r)
    p, rz = z, (r * z).sum()
    res = [r.norm()]
    for _ in range(iters):
        q = S.apply(p)
        a = rz / (p * q).sum()
        x = x + a * p
        r = r - a * q
        res.append(r.norm())
        z = prec(r)
        new = (r * z).sum()
        p, rz = z + (new / rz) * p, new
    return x.reshape(g.shape), torch.stack(res)


def _var64(shape, vx, h, w):
    """Diagonal of the inverse of every block, and minus its log-determinant."""
    S = _system(shape, vx, h, w)
    K = S.K
    var, eye = [], torch.eye(K, dtype=h.dtype, device=h.device)
    for k in range(K):
        e = eye[k].reshape(K, 1, 1, 1).expand(K, *S.dsum.shape)
        var.append(S.precond(e)[k].reshape(-1))
    ld = -2 * sum(torch.log(S.L[k][k]) for k in range(K)).reshape(-1)
    return torch.stack(var), ld


def _start64(prot, means):
    """Constant starting maps from the image means: a shared R2*, the line
    through the non-MT intercepts for A and R1, the MT intercepts for delta."""
    C, te = len(prot["alpha"]), np.array(prot["te"])
    lm = np.log(means)
    sl = [slice(sum(prot["n_echoes"][:c]), sum(prot["n_echoes"][:c + 1])) for c in range(C)]
    num = sum(((te[s] - te[s].mean()) * (lm[s] - lm[s].mean())).sum() for s in sl)
    den = sum(((te[s] - te[s].mean()) ** 2).sum() for s in sl)
    r2 = max(-num / den, 1e-3)
    S0 = [math.exp(lm[s].mean() + r2 * te[s].mean()) for s in sl]
    free = [c for c in range(C) if not prot["mt"][c]]
    X = np.array([S0[c] / math.tan(prot["alpha"][c]) for c in free])
    Y = np.array([S0[c] / math.sin(prot["alpha"][c]) for c in free])
    E = ((X - X.mean()) * (Y - Y.mean())).sum() / ((X - X.mean()) ** 2).sum()
    E = min(max(E, 1e-6), 1 - 1e-6)
    r1 = -math.log(E) / np.mean([prot["tr"][c] for c in free])
    A = (Y.mean() - E * X.mean()) / (1 - E)
    out = [math.log(A), math.log(r1), math.log(r2)]
    if len(free) < C:
        dl = []
        for c in range(C):
            if prot["mt"][c]:
                Ec, a = math.exp(-r1 * prot["tr"][c]), prot["alpha"][c]
                dl.append(1 - S0[c] / (A * math.sin(a) * (1 - Ec) + S0[c] * math.cos(a) * Ec))
        v = min(max(float(np.mean(dl)), 1e-4), 0.5)
        out.append(math.log(v / (1 - v)))
    return out


def _fit64(case, d):
    means = np.array([float(v.double().mean()) for v in d["x"]])
    y0 = torch.tensor([_f32(v) for v in _start64(d["prot"], means)], dtype=torch.float64, device="cuda")
    y = y0[:, None].repeat(1, d["N"])
    F = []
    for it in range(case["gn"] + 1):
        w, e = _jtv64(d, case["vx"], y)
        g, h, nll = _grad_hess64(d, 0, y)
        F.append(float(nll + e))
        if it < case["gn"]:
            y = y - _cg64(d["shape"], case["vx"], h, w, g, y, case["cg"])[0]
    return y, _var64(d["shape"], case["vx"], h, w)[0], F


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        out = []
        for i, t in enumerate(case["shapes"].split(",")):
            out.append(_fit64(case, _subject(case, tuple(int(v) for v in t.split("x")), 1000 * seed + i)))
        return {"y": [o[0] for o in out], "var": [o[1] for o in out], "F": [o[2][-1] for o in out]}
    if kind == "moved":
        d = _moved(case, seed)
        shape, K, prot = d["shape"], d["K"], d["prot"]
        y = d["y"].double()
        T = K * (K + 1) // 2
        g, h = torch.zeros_like(y), torch.zeros((T, d["N"]), dtype=torch.float64, device="cuda")
        nll = 0.0
        for c, A in enumerate(d["affines"]):
            b, f, inside = _cells(shape, A, torch.float64)
            yc = torch.zeros_like(y)
            for w, n in _corners(shape, b, f, inside):
                for k in range(K):
                    yc[k] += w * y[k][n]
            m = torch.nonzero(inside).reshape(-1)
            gc, hc, nc = _contrast64(prot, c, K, d["xs"][c][:, m], yc[:, m], d["b1ps"][c][m].double(),
                                     d["b1ms"][c][m].double(), case["precond"])
            nll = nll + nc
            for w, n in _corners(shape, [v[m] for v in b], [v[m] for v in f], inside[m]):
                for k in range(K):
                    g[k].index_add_(0, n, w * gc[k])
                for t in range(T):
                    h[t].index_add_(0, n, w * hc[t])
        return {"g": g, "h": h, "nll": nll}
    d = _subject(case, _shape(case), seed)
    if kind == "fit":
        y, var, F = _fit64(case, d)
        return {"y": y, "var": var, "F": F}
    if kind == "grad_hess":
        return dict(zip(("g", "h", "nll"), _grad_hess64(d, case["precond"])))
    w, jtv = _jtv64(d, case["vx"])
    if kind == "jtv":
        return {"w": w, "jtv": jtv}
    g, h, _ = _grad_hess64(d, 0)
    g, h, w, y = g.float().double(), h.float().double(), w.float().double(), d["y"].double()
    if kind == "uncertainty":
        var, ld = _var64(d["shape"], case["vx"], h, w)
        s2, r = var[1], y[1]
        mom = torch.stack([torch.exp(r + s2 / 2), torch.expm1(s2) * torch.exp(2 * r + s2),
                           torch.exp(-r + s2 / 2), torch.expm1(s2) * torch.exp(-2 * r + s2)])
        return {"var": var, "logdet": ld, "moments": mom}
    delta, res = _cg64(d["shape"], case["vx"], h, w, g, y, case["cg"], multigrid=kind == "mg")
    return {"delta": delta, "resid": res}
