"""Workloads of the Mueller solver for bodies of revolution, as a user's program calls them.

Every case names a path (``op``), a body, its modes and its options:

  kernels   modal Green's function spectra of (target, source) pairs
  assemble  the weighted matrices of modes 0..M
  lu        batched complex128 LU with partial pivoting
  whole     build + plane-wave data + solve of all modes -M..M, from host geometry to currents
  wave      several bodies built together (one factorization over all their modes), each solved
  rhs       plane-wave data of many incidences on a resident body
  solve     many right-hand sides with the factors of a resident body
  far_grid  far field on a polar x azimuth grid from the modal currents
  eval      fields at points off the surface
"""
from __future__ import annotations

import math
from types import SimpleNamespace

import numpy as np
import torch

import paper_1810_07067_gb300 as mb

DEV = "cuda"
# device blocks that a long-running program keeps between builds (the default cap is below one large body)
CACHE_BYTES = 131 << 30


def listed():
    return [
        # the smallest call: spectra of a handful of pairs (inspection, table generation); latency
        dict(name="kernels_64", op="kernels", pairs=64, M=10, n_phi=64, k0=1.0, k1=1.5, k1i=0.0),
        # the smallest body of the tests: a unit sphere in complex128, default precision, both polarisations
        dict(name="sphere_fp64", op="whole", body="sphere", panels=4, M=10, n_phi=64, k0=1.0, k1=1.5, k1i=0.0,
             precision=0, formulation=0, nrhs=2),
        # an edge-refined lossy cylinder in complex128 throughout
        dict(name="cylinder_fp64", op="whole", body="cylinder", panels=20, M=64, n_phi=256, k0=5.0, k1=7.5,
             k1i=0.01, precision=0, formulation=0, nrhs=4),
        # the full-size lossy cylinder, mixed precision, 8 incidences x 2 polarisations
        dict(name="cylinder_mixed", op="whole", body="cylinder", panels=36, M=64, n_phi=256, k0=5.0, k1=7.5,
             k1i=0.01, precision=1, formulation=0, nrhs=16),
        # the headline body: smooth random curve, 1024 nodes, modes -128..128, mixed precision
        dict(name="random_mixed", op="whole", body="random", panels=64, M=128, n_phi=512, k0=10.0, k1=15.0, k1i=0.0,
             precision=1, formulation=0, nrhs=2),
        # part of the batched workload: bodies of different sizes factored together, odd mode counts
        dict(name="wave_mixed", op="wave", bodies=6, panels=13, panels_hi=24, M=32, M_hi=60, k0=3.0, precision=1,
             nrhs=2),
        # matrices only, of a closed curve, in the indirect form
        dict(name="torus_assemble", op="assemble", body="torus", panels=20, M=33, n_phi=128, k0=2.0, k1=3.0, k1i=0.0,
             formulation=1),
        # dense factorization alone, a ragged order
        dict(name="lu_fp64", op="lu", n=1250, batch=9),
        # serving: one request's incidences turned into modal data ...
        dict(name="rhs_waves", op="rhs", body="random", panels=32, M=64, k0=6.0, k1=9.0, k1i=0.0, nrhs=96),
        # ... solved with the resident factors ...
        dict(name="solve_many", op="solve", body="random", panels=32, M=64, k0=6.0, k1=9.0, k1i=0.0, precision=1,
             nrhs=96),
        # ... and its bistatic pattern on a one-degree grid
        dict(name="far_grid", op="far_grid", body="random", panels=32, M=64, k0=6.0, k1=9.0, k1i=0.0, nrhs=8,
             polar=180, azim=360),
        # fields at observation points outside the body
        dict(name="eval_points", op="eval", body="cylinder", panels=20, M=32, k0=5.0, k1=7.5, k1i=0.01, nrhs=2,
             targets=100, region=0),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["kernels", "whole", "whole", "wave", "assemble", "lu", "rhs", "solve", "far_grid", "eval"])
    body = rng.choice(["sphere", "cylinder", "cone", "random", "torus"])
    k0 = round(rng.uniform(1.0, 8.0), 3)
    k1 = round(1.5 * k0, 3)
    k1i = rng.choice([0.0, 0.0, 0.01])
    med = dict(k0=k0, k1=k1, k1i=k1i)
    if op == "kernels":
        return dict(op=op, pairs=_logint(rng, 16, 20000), M=rng.randint(4, 80), n_phi=rng.choice([64, 128, 256]), **med)
    if op == "lu":
        n = _logint(rng, 64, 1800)
        return dict(op=op, n=n, batch=max(1, min(_logint(rng, 1, 64), int(3e10 / n ** 3))))
    if op == "wave":
        lo = rng.randint(6, 14)
        M = rng.randint(12, 40)
        return dict(op=op, bodies=rng.randint(2, 6), panels=lo, panels_hi=lo + rng.randint(1, 8), M=M,
                    M_hi=M + rng.randint(1, 16), k0=round(rng.uniform(1.0, 6.0), 3), precision=rng.choice([0, 1, 1]),
                    nrhs=rng.randint(1, 3))
    precision = rng.choice([0, 1, 1, 2])
    panels = _logint(rng, 4, 22 if precision == 0 else 40)
    M = _logint(rng, 4, 60)
    if op == "assemble":
        return dict(op=op, body=body, panels=min(panels, 24), M=M, n_phi=16, formulation=rng.choice([0, 1]), **med)
    if op == "whole":
        return dict(op=op, body=body, panels=panels, M=M, n_phi=16, precision=precision,
                    formulation=rng.choice([0, 0, 1]), nrhs=_logint(rng, 1, 16), **med)
    panels = min(panels, 32)
    if op == "rhs":
        return dict(op=op, body=body, panels=panels, M=M, nrhs=_logint(rng, 1, 200), **med)
    if op == "solve":
        return dict(op=op, body=body, panels=panels, M=M, precision=precision, nrhs=_logint(rng, 1, 128), **med)
    if op == "far_grid":
        return dict(op=op, body=body, panels=panels, M=M, nrhs=rng.randint(1, 8), polar=_logint(rng, 9, 180),
                    azim=_logint(rng, 9, 360), **med)
    return dict(op=op, body=body, panels=min(panels, 24), M=M, nrhs=rng.randint(1, 4), targets=_logint(rng, 1, 128),
                region=rng.choice([0, 0, 1]), **med)


# ---------------------------------------------------------------- inputs
def _sample(edges, fun, closed=False):
    """A generating curve t -> (r, z, r', z') at the 16 Gauss points of each panel."""
    x, _ = np.polynomial.legendre.leggauss(16)
    out = [], [], [], []
    for a, b in zip(edges[:-1], edges[1:]):
        r, z, dr, dz = fun(0.5 * (a + b) + 0.5 * (b - a) * x)
        for o, v in zip(out, (r, z, 0.5 * (b - a) * dr, 0.5 * (b - a) * dz)):
            o.append(v)
    r, z, dr, dz = (np.concatenate(o) for o in out)
    return SimpleNamespace(n_panels=len(edges) - 1, r=r, z=z, dr=dr, dz=dz, closed=closed)


def _polyline(verts, base, corners, panels):
    """Straight segments with base[i] equal panels each; the panels at the given (segment, end)
    corners are halved toward them, level by level, until the curve has about `panels` panels."""
    levels = max(1, round((panels - sum(base)) / len(corners)))
    edges, pts = [0.0], []
    for s, nb in enumerate(base):
        cuts = list(np.linspace(0.0, 1.0, nb + 1))
        if (s, 0) in corners:
            cuts += [cuts[1] / 2 ** (q + 1) for q in range(levels)]
        if (s, 1) in corners:
            w = 1.0 - cuts[nb - 1]
            cuts += [1.0 - w / 2 ** (q + 1) for q in range(levels)]
        edges += [s + c for c in sorted(cuts)[1:]]
        pts.append((verts[s], verts[s + 1]))

    def fun(t):
        s = min(int(t[0]), len(pts) - 1)
        (ra, za), (rb, zb) = pts[s]
        u, one = t - s, np.ones_like(t)
        return ra + (rb - ra) * u, za + (zb - za) * u, (rb - ra) * one, (zb - za) * one
    return _sample(edges, fun)


def _curve(body, panels, rng):
    """A body of about unit size; its shape parameters come from rng."""
    if body == "cylinder":
        R, h = rng.uniform(0.97, 1.0), rng.uniform(0.95, 1.05)
        return _polyline([(0, -h), (R, -h), (R, h), (0, h)], (2, 4, 2), {(0, 1), (1, 0), (1, 1), (2, 0)}, panels)
    if body == "cone":
        R, h = rng.uniform(0.97, 1.0), rng.uniform(0.95, 1.05)
        return _polyline([(0, -h), (R, -h), (0, h)], (2, 4), {(0, 1), (1, 0), (1, 1)}, panels)
    if body == "torus":
        n, R, b = max(panels, 4), rng.uniform(1.95, 2.0), rng.uniform(0.48, 0.52)
        return _sample(np.linspace(0, 2 * np.pi, n + 1),
                       lambda t: (R + np.cos(t), b * np.sin(t), -np.sin(t), b * np.cos(t)), True)
    j = np.arange(1, 7)
    a = rng.uniform(-0.08, 0.08, 6) if body == "random" else np.zeros(6)
    c = 1.0 if body == "random" else rng.uniform(0.97, 1.0)

    def fun(t):
        s = c + np.cos(np.outer(t, j)) @ a
        ds = -np.sin(np.outer(t, j)) @ (a * j)
        return np.sin(t) * s, -c * np.cos(t), np.cos(t) * s + np.sin(t) * ds, c * np.sin(t)
    return _sample(np.linspace(0, np.pi, panels + 1), fun)


def _media(c):
    eps1 = (complex(c["k1"], c["k1i"]) / c["k0"]) ** 2
    return SimpleNamespace(omega=c["k0"], eps0=1.0, mu0=1.0, eps1=eps1, mu1=1.0)


def _waves(rng, n):
    d = rng.normal(size=(n, 3))
    d /= np.linalg.norm(d, axis=1, keepdims=True)
    e = np.cross(d, rng.normal(size=(n, 3)))
    return d, e / np.linalg.norm(e, axis=1, keepdims=True)


def _currents(c, N, seed):
    """Modal currents whose modes fall off as those of an incident wave do beyond k0 r."""
    g = torch.Generator(device=DEV).manual_seed(int(seed))
    x = torch.randn((2 * c["M"] + 1, c["nrhs"], 4 * N), dtype=torch.complex128, device=DEV, generator=g)
    m = torch.arange(-c["M"], c["M"] + 1, device=DEV, dtype=torch.float64).abs()
    return x * torch.exp(-0.7 * (m - c["k0"]).clamp(min=0))[:, None, None]


def _targets(c, rng):
    n = c["targets"]
    u = _waves(rng, n)[0]
    if c["region"] == 0:
        return u * rng.uniform(4.0, 8.0, (n, 1))
    if c["body"] == "torus":  # inside the tube, around its centre circle
        phi = rng.uniform(0, 2 * np.pi, n)
        return np.stack([2 * np.cos(phi), 2 * np.sin(phi), np.zeros(n)], 1) + 0.05 * u
    return np.array([0.0, 0.0, -0.2]) + 0.1 * u


def _options(c):
    return mb.Options(n_phi=c.get("n_phi", 16), formulation=c.get("formulation", 0), precision=c.get("precision", 0))


def _pairs(c, rng):
    """Targets and sources on a body's meridian: most well apart, one in eight within a tenth."""
    n = c["pairs"]
    rt, zt = rng.uniform(0.3, 1.2, n), rng.uniform(-1.0, 1.0, n)
    ang = rng.uniform(0, 2 * np.pi, n)
    d = np.where(rng.uniform(size=n) < 0.125, np.exp(rng.uniform(np.log(0.02), np.log(0.1), n)), rng.uniform(0.1, 1.0, n))
    rs = rt + d * np.cos(ang)
    rs = np.where(rs < 0.05, rt + d * np.abs(np.cos(ang)) + 0.05, rs)
    return np.stack([rt, zt, rs, zt + d * np.sin(ang)], 1)


def prepare(case, seed):
    c, rng = dict(case), np.random.default_rng(int(seed))
    mb.cache_limit(CACHE_BYTES)
    s = SimpleNamespace(c=c)
    op = c["op"]
    if op == "kernels":
        s.pairs = _pairs(c, rng)
        s.out = torch.empty((c["pairs"], 9, c["M"] + 2), dtype=torch.complex128, device=DEV)
        return s
    if op == "lu":
        g = torch.Generator(device=DEV).manual_seed(int(seed))
        s.A0 = torch.randn((c["batch"], c["n"], c["n"]), dtype=torch.complex128, device=DEV, generator=g)
        s.A = torch.empty_like(s.A0)
        s.piv = torch.empty((c["batch"], c["n"]), dtype=torch.int32, device=DEV)
        s.info = torch.empty((c["batch"],), dtype=torch.int32, device=DEV)
        return s
    if op == "wave":
        s.bodies = []
        for q in range(c["bodies"]):  # sizes spread over the wave's range
            f = q / max(1, c["bodies"] - 1)
            P, M = round(c["panels"] + f * (c["panels_hi"] - c["panels"])), round(c["M"] + f * (c["M_hi"] - c["M"]))
            k0 = c["k0"] * (1 + 0.1 * q)
            s.bodies.append((_curve("random", P, rng), _media(dict(k0=k0, k1=1.5 * k0, k1i=0.0)), M))
        s.dirs, s.pols = _waves(rng, c["nrhs"])
        return s
    s.curve, s.media = _curve(c["body"], c["panels"], rng), _media(c)
    N = 16 * s.curve.n_panels
    if op == "assemble":
        s.A = torch.empty((c["M"] + 1, 4 * N, 4 * N), dtype=torch.complex128, device=DEV)
    elif op == "eval":
        s.targets = _targets(c, rng)
        s.x = _currents(c, N, seed)
        s.out = torch.empty((c["nrhs"], c["targets"], 6), dtype=torch.complex128, device=DEV)
    elif op == "far_grid":
        s.x = _currents(c, N, seed)
        s.E = torch.empty((c["nrhs"], c["polar"], c["azim"], 3), dtype=torch.complex128, device=DEV)
    else:
        s.dirs, s.pols = _waves(rng, c["nrhs"])
        s.rhs = torch.empty((2 * c["M"] + 1, c["nrhs"], 4 * N), dtype=torch.complex128, device=DEV)
        s.x = torch.empty_like(s.rhs)
    if op in ("rhs", "solve", "far_grid", "eval"):  # the resident body
        s.ctx = mb.build(s.curve, s.media, c["M"], mb.Options(n_phi=16, precision=c.get("precision", 1)))
        if op == "solve":
            s.ctx.rhs_planewave(s.dirs, s.pols, s.rhs)
    return s


def run(s):
    c = s.c
    op = c["op"]
    if op == "kernels":
        return mb.modal_kernels(s.pairs, c["k0"], complex(c["k1"], c["k1i"]), c["M"], c["n_phi"], s.out)
    if op == "lu":
        s.A.copy_(s.A0)
        mb.lu_batched(s.A, s.piv, s.info)
        return s.A, s.piv, s.info
    if op == "assemble":
        return mb.assemble(s.curve, s.media, c["M"], s.A, _options(c))
    if op == "whole":
        ctx = mb.build(s.curve, s.media, c["M"], _options(c))
        ctx.rhs_planewave(s.dirs, s.pols, s.rhs)
        ctx.solve(s.rhs, s.x)
        ctx.close()
        return s.x
    if op == "wave":
        out = []
        for ctx in mb.build_many(s.bodies, mb.Options(n_phi=16, precision=c["precision"])):
            rhs = torch.empty((2 * ctx.M + 1, c["nrhs"], 4 * ctx.N), dtype=torch.complex128, device=DEV)
            x = torch.empty_like(rhs)
            ctx.rhs_planewave(s.dirs, s.pols, rhs)
            ctx.solve(rhs, x)
            ctx.close()
            out.append(x)
        return out
    if op == "rhs":
        return s.ctx.rhs_planewave(s.dirs, s.pols, s.rhs)
    if op == "solve":
        return s.ctx.solve(s.rhs, s.x)
    if op == "far_grid":
        return s.ctx.far_field_grid(s.x, s.E)
    return s.ctx.eval(s.x, s.targets, c["region"], s.out)


# ---------------------------------------------------------------- work
def _nodes(c):
    return 16 * _curve(c["body"], c["panels"], np.random.default_rng(0)).n_panels


def _body_work(N, M, nrhs):
    """Assembly (per node pair: samples of nine kernels over the ring, their cosine transform, a 4 x 4 block per
    mode), LU of M + 1 systems of order 4N and the substitutions of 2M + 1 modes; the matrices written once."""
    n, ring = 4 * N, 2 * M + 64
    flops = N * N * (ring // 2 * 140 + 9 * 2.5 * ring * math.log2(ring) + 256 * (M + 1))
    flops += (M + 1) * 8 / 3 * n ** 3 + 8.0 * n * n * (2 * M + 1) * nrhs
    return 16.0 * (M + 1) * n * n + 32.0 * (2 * M + 1) * nrhs * n, flops


def work(case):
    c = case
    op = c["op"]
    if op == "kernels":
        ring = max(c["n_phi"], 2 * c["M"] + 4)
        f = c["pairs"] * (ring // 2 * 140 + 9 * 2.5 * ring * math.log2(ring))
        return {"bytes": c["pairs"] * (32 + 9 * (c["M"] + 2) * 16), "flops": f}
    if op == "lu":
        return {"bytes": 32.0 * c["batch"] * c["n"] ** 2, "flops": c["batch"] * 8 / 3 * c["n"] ** 3}
    if op == "wave":
        b = f = 0.0
        for q in range(c["bodies"]):
            g = q / max(1, c["bodies"] - 1)
            bb, ff = _body_work(16 * round(c["panels"] + g * (c["panels_hi"] - c["panels"])),
                                round(c["M"] + g * (c["M_hi"] - c["M"])), c["nrhs"])
            b, f = b + bb, f + ff
        return {"bytes": b, "flops": f}
    N, M = _nodes(c), c["M"]
    n, modes = 4 * N, 2 * M + 1
    if op == "whole":
        b, f = _body_work(N, M, c["nrhs"])
        return {"bytes": b, "flops": f}
    if op == "assemble":
        b, f = _body_work(N, M, 0)
        return {"bytes": b, "flops": f - (M + 1) * 8 / 3 * n ** 3}
    if op == "rhs":
        ring = 2 * M + 64
        return {"bytes": 16.0 * modes * c["nrhs"] * n,
                "flops": c["nrhs"] * N * (ring * 60 + 4 * 5 * ring * math.log2(ring))}
    if op == "solve":  # the factors once, two vectors each way
        return {"bytes": (8.0 if c["precision"] else 16.0) * (M + 1) * n * n + 32.0 * modes * c["nrhs"] * n,
                "flops": 8.0 * n * n * modes * c["nrhs"]}
    if op == "far_grid":
        return {"bytes": 16.0 * modes * c["nrhs"] * n + 48.0 * c["nrhs"] * c["polar"] * c["azim"],
                "flops": 8.0 * 8 * c["nrhs"] * c["polar"] * modes * N +
                c["nrhs"] * c["polar"] * 3 * 5 * c["azim"] * math.log2(max(c["azim"], 2))}
    ring = 2 * M + 64
    return {"bytes": 16.0 * modes * c["nrhs"] * n + 96.0 * c["nrhs"] * c["targets"],
            "flops": c["nrhs"] * N * ring * (c["targets"] * 250 + 4 * 5 * math.log2(ring))}


# ---------------------------------------------------------------- exact values in 64 bits
def _exact_kernels(c, rng):
    p = torch.from_numpy(_pairs(c, rng)).to(DEV)
    M, ks = c["M"], (complex(c["k0"]), complex(c["k1"], c["k1i"]))
    x, w = np.polynomial.legendre.leggauss(32)
    nodes, weights = [], []  # graded toward phi = 0, where close pairs peak
    top = math.pi
    for lev in range(14):
        lo = 0.0 if lev == 13 else top / 2
        sub = max(1, math.ceil((top - lo) * (M + 2 + 3 * abs(ks[1])) / 12))
        for q in range(sub):
            a, b = lo + (top - lo) * q / sub, lo + (top - lo) * (q + 1) / sub
            nodes.append(0.5 * (a + b) + 0.5 * (b - a) * x)
            weights.append((b - a) * w)  # twice the half range
        top = lo
    phi = torch.from_numpy(np.concatenate(nodes)).to(DEV)
    T = torch.cos(phi[:, None] * torch.arange(M + 2, device=DEV)) * torch.from_numpy(np.concatenate(weights)).to(DEV)[:, None]
    s2 = torch.sin(phi / 2) ** 2
    out = torch.empty((len(p), 9, M + 2), dtype=torch.complex128, device=DEV)
    for lo in range(0, len(p), 1024):
        rt, zt, rs, zs = (v[:, None] for v in p[lo:lo + 1024].T)
        dr, dz = rt - rs, zt - zs
        rho = torch.sqrt(dr ** 2 + dz ** 2 + 4 * rt * rs * s2)
        rd = dr + 2 * rs * s2
        E = []
        for k in ks:
            q = 1j * k * rho
            e = torch.exp(q) / (4 * math.pi)
            E.append((e / rho, e * (q - 1) / (2 * rho ** 3), e * (q * q - 3 * q + 3) / (4 * rho ** 5)))
        d1, d2 = E[0][1] - E[1][1], E[0][2] - E[1][2]
        F = [E[0][0], E[1][0], 2 * rd * E[0][1], 2 * dz * E[0][1], 2 * rd * E[1][1], 2 * dz * E[1][1],
             4 * rd ** 2 * d2 + 2 * d1, 4 * rd * dz * d2, 4 * dz ** 2 * d2 + 2 * d1]
        F = torch.stack(F, 1)
        out[lo:lo + 1024] = torch.complex(F.real @ T, F.imag @ T)
    return out


def _exact_lu(c, seed):
    """Right-looking LU by blocks of 64 columns; pivot: the largest |a|, the first row of equals."""
    g = torch.Generator(device=DEV).manual_seed(int(seed))
    n, B = c["n"], c["batch"]
    A = torch.randn((B, n, n), dtype=torch.complex128, device=DEV, generator=g).transpose(1, 2).contiguous()
    piv = torch.zeros((B, n), dtype=torch.int32, device=DEV)
    idx = torch.arange(B, device=DEV)
    for k0 in range(0, n, 64):
        k1 = min(n, k0 + 64)
        for k in range(k0, k1):
            col = A[:, k:, k]
            p = k + torch.argmax(col.real ** 2 + col.imag ** 2, 1)
            piv[:, k] = p.int()
            a, b = A[:, k].clone(), A[idx, p].clone()
            A[idx, p], A[:, k] = a, b
            A[:, k + 1:, k] /= A[:, k, k][:, None]
            A[:, k + 1:, k + 1:k1] -= A[:, k + 1:, k, None] * A[:, k, None, k + 1:k1]
        if k1 < n:
            U = torch.linalg.solve_triangular(A[:, k0:k1, k0:k1], A[:, k0:k1, k1:], upper=False, unitriangular=True)
            A[:, k0:k1, k1:] = U
            A[:, k1:, k1:] -= A[:, k1:, k0:k1] @ U
    return A.transpose(1, 2).contiguous(), piv, torch.zeros((B,), dtype=torch.int32, device=DEV)


def _geometry(cv):
    sp = np.hypot(cv.dr, cv.dz)
    w = np.tile(np.polynomial.legendre.leggauss(16)[1], cv.n_panels) * sp
    return [torch.from_numpy(np.ascontiguousarray(v)).to(DEV) for v in (cv.r, cv.z, cv.dr / sp, cv.dz / sp, w)]


def _exact_rhs(c, rng):
    r, z, rp, zp, _ = _geometry(_curve(c["body"], c["panels"], rng))
    dirs, pols = _waves(rng, c["nrhs"])
    M, k0, N = c["M"], c["k0"], len(r)
    nt = 1 << math.ceil(math.log2(2 * (2 * M + 4 * k0 * float(r.max()) + 64)))
    th = torch.arange(nt, dtype=torch.float64, device=DEV) * (2 * math.pi / nt)
    ct, st = torch.cos(th), torch.sin(th)
    modes = torch.arange(-M, M + 1, device=DEV) % nt
    out = torch.empty((2 * M + 1, c["nrhs"], N, 4), dtype=torch.complex128, device=DEV)
    for q in range(c["nrhs"]):
        d, e = dirs[q], pols[q]
        ph = torch.exp(1j * k0 * (r[:, None] * (d[0] * ct + d[1] * st) + z[:, None] * d[2]))
        for f, v in ((0, e), (2, np.cross(d, e))):  # H: k0 / (omega mu0) = 1
            vt = rp[:, None] * (v[0] * ct + v[1] * st) + zp[:, None] * v[2]
            vth = v[1] * ct - v[0] * st
            for a, t in ((f, vth * ph), (f + 1, -vt * ph)):
                out[:, q, :, a] = (1j * k0 / nt) * torch.fft.fft(t, dim=1)[:, modes].T
    return out.reshape(2 * M + 1, c["nrhs"], 4 * N)


def _exact_far_grid(c, rng, seed):
    r, z, rp, zp, w = _geometry(_curve(c["body"], c["panels"], rng))
    M, k0, N = c["M"], c["k0"], len(r)
    x = _currents(c, N, seed).reshape(2 * M + 1, c["nrhs"], N, 4)
    na = 1 << math.ceil(math.log2(2 * (2 * M + 4 * k0 * float(r.max()) + 64)))
    al = torch.arange(na, dtype=torch.float64, device=DEV) * (2 * math.pi / na)
    ca, sa = torch.cos(al), torch.sin(al)
    modes = (-torch.arange(-M, M + 1, device=DEV)) % na  # ring integrals against e^{+i m alpha}
    phi = torch.arange(c["azim"], dtype=torch.float64, device=DEV) * (2 * math.pi / c["azim"])
    em = torch.exp(1j * (phi[:, None] * torch.arange(-M, M + 1, device=DEV)))
    out = torch.empty((c["nrhs"], c["polar"], c["azim"], 3), dtype=torch.complex128, device=DEV)
    for p in range(c["polar"]):
        t = (p + 0.5) * math.pi / c["polar"]
        sth, cth = math.sin(t), math.cos(t)
        f = torch.exp(-1j * k0 * sth * r[:, None] * ca)
        I0, Ic, Is = (torch.fft.fft(f * g, dim=1)[:, modes].T * (2 * math.pi / na) for g in (torch.ones_like(ca), ca, sa))
        ph = w * r * torch.exp(-1j * k0 * cth * z)
        V = []
        for a in (0, 2):
            u, v = x[..., a] * ph, x[..., a + 1] * ph
            V.append([torch.einsum("mqn,mn->mq", u, rp * Ic) - torch.einsum("mqn,mn->mq", v, Is),
                      torch.einsum("mqn,mn->mq", u, rp * Is) + torch.einsum("mqn,mn->mq", v, Ic),
                      torch.einsum("mqn,mn->mq", u, zp * I0)])
        J, K = V
        xJ = sth * J[0] + cth * J[2]
        X = (-cth * K[1], cth * K[0] - sth * K[2], sth * K[1])
        F = [(1j * k0 * (J[a] - h * xJ) + 1j * k0 * X[a]) / (4 * math.pi) for a, h in enumerate((sth, 0.0, cth))]
        E = [(em @ v).T for v in F]  # [nrhs, azim]
        out[:, p] = torch.stack([torch.cos(phi) * E[0] - torch.sin(phi) * E[1],
                                 torch.sin(phi) * E[0] + torch.cos(phi) * E[1], E[2]], -1)
    return out


def _exact_eval(c, rng, seed):
    r, z, rp, zp, w = _geometry(_curve(c["body"], c["panels"], rng))
    X = torch.from_numpy(_targets(c, rng)).to(DEV)
    near = torch.hypot(torch.hypot(X[:, 0], X[:, 1])[:, None] - r, X[:, 2, None] - z).amin(0).reshape(-1, 16).amin(1)
    if bool((1.5 * w.reshape(-1, 16).sum(1) > near).any()):
        return None  # close targets are summed over refined panels, with interpolated currents
    M, N, om = c["M"], len(r), c["k0"]
    x = _currents(c, N, seed).reshape(2 * M + 1, c["nrhs"], N, 4)
    k = complex(om) if c["region"] == 0 else complex(c["k1"], c["k1i"])
    eps, sg = (1.0, 1.0) if c["region"] == 0 else ((k / om) ** 2, -1.0)
    nt = 2 * (2 * M + 2 * math.ceil(abs(k) * float(r.max())) + 128)
    th = torch.arange(nt, dtype=torch.float64, device=DEV) * (2 * math.pi / nt)
    ct, st, one = torch.cos(th), torch.sin(th), torch.ones_like(th)
    em = torch.exp(1j * (th[:, None] * torch.arange(-M, M + 1, device=DEV)))
    y = torch.stack([r[:, None] * ct, r[:, None] * st, z[:, None] * one], -1).reshape(-1, 3)
    da = (w * r * (2 * math.pi / nt)).repeat_interleave(nt)
    tang = torch.stack([rp[:, None] * ct, rp[:, None] * st, zp[:, None] * one], -1)
    eth = torch.stack([-st, ct, 0 * one], -1)[None]
    out = torch.empty((c["nrhs"], len(X), 6), dtype=torch.complex128, device=DEV)
    for q in range(c["nrhs"]):
        cur = torch.einsum("tm,mna->nta", em, x[:, q])
        V = [(cur[..., a, None] * tang + cur[..., a + 1, None] * eth).reshape(-1, 3) for a in (0, 2)]
        for i in range(len(X)):
            R3 = X[i] - y
            R = R3.norm(dim=1)
            h = R3 / R[:, None]
            G = da * torch.exp(1j * k * R) / (4 * math.pi * R)
            c1 = (G * (1j * k - 1 / R))[:, None]
            aa, bb = (G * (k * k + 1j * k / R - 1 / R ** 2))[:, None], (G * (3 / R ** 2 - k * k - 3j * k / R))[:, None]
            hc = h.to(torch.complex128)
            cc = [(aa * v + bb * (hc * v).sum(1, keepdim=True) * hc).sum(0) for v in V]
            cu = [(c1 * torch.linalg.cross(hc, v)).sum(0) for v in V]
            out[q, i, :3] = -sg / (1j * om * eps) * cc[0] + sg * cu[1]
            out[q, i, 3:] = sg / (1j * om) * cc[1] + sg * cu[0]
    return out


def exact(case, seed):
    """Where plain 64-bit torch gives the outputs in seconds; None for what needs a whole assembly."""
    c, rng = dict(case), np.random.default_rng(int(seed))
    op = c["op"]
    if op == "kernels":
        return _exact_kernels(c, rng)
    if op == "lu":
        return _exact_lu(c, seed)
    if op == "rhs":
        return _exact_rhs(c, rng)
    if op == "far_grid":
        return _exact_far_grid(c, rng, seed)
    if op == "eval":
        return _exact_eval(c, rng, seed)
    return None
