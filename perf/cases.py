"""Performance cases of the multibody scattering solver: what a program that uses it runs.

A scattering program describes its bodies once, builds the scattering matrices of their
shapes, and then works with many incident fields: every GMRES iteration applies the
inter-body sum B and the block-diagonal inverse D^{-1}, in single precision inside the
mixed solve, in FP64 or double-float for the residual; after the solve it asks for the
far field.  So most cases are one operator through its public call, on the geometries of
`workloads/` or shapes like them; two are whole solves and one is the far field.

Results of the single-precision operators are handed on as complex64, the precision they
are computed in; every other result is complex128.

A case is a dict of
  op      "sum" (B sigma), "dinv" (D^{-1} y), "apply" (sigma + D^{-1} B sigma), "solve", "far"
  prec    "f64", "f32", "df" (double-float); a solve's "mixed" (double-float residual) or "f64"
  geo     "spheres", "spheroids", "slender", "shells", "uneven" (see bodies_of)
  bodies, panels, gl, modes: the discretisation of a body: panels x gl rings of `modes` nodes
  k       wavenumber (eta = k)
  rhs     right-hand sides in one call
  eps     tolerance of the skeletons of the accelerated scheme (0: the direct solve)
  points  directions of the far field (0: none)
"""
import math

import numpy as np
import torch

from paper_1406_0236_gb300 import (HZB_OPEN_SHELL, HZB_PREC_DOUBLE_FLOAT, HZB_PREC_FP64, HZB_PREC_MIXED_FP32,
                                   HZB_SPHERE, HZB_SPHEROID, Options, Solver)

PREC = {"f64": HZB_PREC_FP64, "f32": HZB_PREC_MIXED_FP32, "df": HZB_PREC_DOUBLE_FLOAT}


def case(name, op, prec, geo, bodies, panels, gl, modes, k, rhs, eps=0.0, points=0):
    return {"name": name, "op": op, "prec": prec, "geo": geo, "bodies": bodies, "panels": panels, "gl": gl,
            "modes": modes, "k": k, "rhs": rhs, "eps": eps, "points": points}


def listed():
    return [
        # the smallest call: one FP64 operator apply on 432 unknowns, all launches and latency
        case("apply_f64_432", "apply", "f64", "spheres", 2, 4, 6, 9, 1.0, 1),
        # one inner GMRES apply of the two-sphere workload, one right-hand side
        case("apply_f32_8200", "apply", "f32", "spheres", 2, 10, 10, 41, 2.0, 1),
        # the inner inter-body sum of the headline workload: eight spheroids, 258,560 unknowns
        case("sum_f32_258560", "sum", "f32", "spheroids", 8, 20, 16, 101, 4.0, 1),
        # the inner sum of a batched solve on sphere, spheroid and open shells
        case("sum_f32_29280_r16", "sum", "f32", "shells", 4, 12, 10, 61, 6.0, 16),
        # the refinement residual's sum, one right-hand side and a batch
        case("sum_df_29280", "sum", "df", "shells", 4, 12, 10, 61, 6.0, 1),
        case("sum_df_8200_r64", "sum", "df", "spheres", 2, 10, 10, 41, 2.0, 64),
        # the library's default precision on a mid-sized geometry
        case("sum_f64_29280", "sum", "f64", "shells", 4, 12, 10, 61, 6.0, 1),
        # the block-diagonal inverse of a batched inner solve at full size
        case("dinv_f32_258560_r16", "dinv", "f32", "spheroids", 8, 20, 16, 101, 4.0, 16),
        # uneven bodies, odd sizes: the residual operator of a small batch
        case("apply_df_uneven_r8", "apply", "df", "uneven", 3, 12, 8, 41, 4.0, 8),
        # whole calls: 64 plane waves at once (a batch of the warm start's training set), and
        # four through the accelerated scheme
        case("solve_mixed_8200_r64", "solve", "mixed", "spheres", 2, 10, 10, 41, 2.0, 64),
        case("solve_accel_21960_r4", "solve", "mixed", "slender", 3, 12, 10, 61, 2.0, 4, eps=1e-8),
        # the far field of that batch over a sphere of directions
        case("far_8200_r64", "far", "f64", "spheres", 2, 10, 10, 41, 2.0, 64, points=512),
    ]


# seconds of one pass, roughly: per ordered pair of nodes, per right-hand side beyond the first
_PAIR = {"f32": 8e-13, "df": 8e-12, "f64": 5e-11}
_MORE = {"f32": 0.06, "df": 0.2, "f64": 0.2}


def draw(rng):
    """Another operator call, solve or far field, sizes over the whole range."""
    op = rng.choice(["sum", "sum", "sum", "dinv", "apply", "apply", "solve", "far"])
    prec = "f64" if op == "far" else "mixed" if op == "solve" else rng.choice(["f32", "f32", "df", "f64"])
    geo = rng.choice(["spheres", "spheroids", "shells", "uneven"])
    bodies = 3 if geo == "uneven" else rng.choice([2, 3, 4, 5, 8])
    if op in ("solve", "far"):
        rhs, top = rng.choice([1, 2, 5, 16, 33, 64]), 9000
    else:
        rhs = rng.choice({"f32": [1, 1, 2, 3, 6, 8, 16, 24, 33, 64], "df": [1, 1, 2, 4, 7, 8, 16, 32, 64],
                          "f64": [1, 1, 2, 3, 4, 8, 9]}[prec])
        # at most about 25 ms of pair work, and 100,000 unknowns x right-hand sides x 16
        top = min(math.sqrt(0.025 / (_PAIR[prec] * (1 + _MORE[prec] * (rhs - 1)))), 1.6e6 / rhs, 150000)
    n = math.exp(rng.uniform(math.log(450.0), math.log(max(top, 900.0)))) / bodies
    rings = math.sqrt(n * rng.uniform(1.2, 3.0))
    gl = rng.choice([6, 7, 8, 10, 13, 16])
    panels = max(9 if geo == "shells" else 5, min(24, round(rings / gl)))
    modes = 2 * (max(9, min(121, round(n / (panels * gl)))) // 2) + 1
    if geo == "uneven":
        modes = max(modes, 17)
    return {"op": op, "prec": prec, "geo": geo, "bodies": bodies, "panels": panels, "gl": gl, "modes": modes,
            "k": round(rng.uniform(1.0, 4.0), 2), "rhs": rhs, "eps": 0.0,
            "points": rng.choice([7, 64, 361]) if op == "far" else 0}


# ------------------------------------------------------------------ geometry

def rotation(axis):
    """The smallest rotation taking e_z to the direction of `axis`."""
    a = np.asarray(axis, float) / np.linalg.norm(axis)
    if a[2] < -1.0 + 1e-12:
        return np.diag([1.0, -1.0, -1.0])
    v = np.array([-a[1], a[0], 0.0])
    vx = np.array([[0.0, -v[2], v[1]], [v[2], 0.0, -v[0]], [-v[1], v[0], 0.0]])
    return np.eye(3) + vx + vx @ vx / (1.0 + a[2])


def bodies_of(c):
    """(kind, params, panels, gl, modes, centre, rotation) of every body of the case.

    spheres: unit spheres on a line, 3 apart.  spheroids: semi-axes (1, 1, 2), turned at
    random, on a grid of spacing 5.  slender: semi-axes (1/2, 1/2, 1) on a line, 3.5 apart,
    for the accelerated scheme.  shells: sphere, spheroid and two thick open shells in turn
    on a grid of spacing 4.5.  uneven: a sphere and two spheroids of different sizes and
    discretisations on a line, 5 apart."""
    rng = np.random.default_rng(20140601)
    nb, geo = c["bodies"], c["geo"]
    side = 2 if nb <= 8 else 3
    out = []
    for q in range(nb):
        turn = rotation(rng.standard_normal(3))
        grid = np.array([q % side, q // side % side, q // side ** 2], float) - 0.5 * (side - 1)
        panels, modes = c["panels"], c["modes"]
        if geo == "spheres":
            kind, par, cen, turn = HZB_SPHERE, (1.0,), np.array([3.0 * (q - 0.5 * (nb - 1)), 0.0, 0.0]), np.eye(3)
        elif geo == "spheroids":
            kind, par, cen = HZB_SPHEROID, (1.0, 2.0), 5.0 * grid
        elif geo == "slender":
            kind, par, cen = HZB_SPHEROID, (0.5, 1.0), np.array([3.5 * q, 0.4 * (q % 2), 0.0])
        elif geo == "shells":
            kind, par = [(HZB_SPHERE, (1.0,)), (HZB_SPHEROID, (1.0, 2.0)),
                         (HZB_OPEN_SHELL, (1.0, 0.8, np.pi / 3.0, 0.1)),
                         (HZB_OPEN_SHELL, (1.0, 0.8, np.pi / 3.0, 0.1))][q % 4]
            cen = 4.5 * grid
        else:
            kind, par = [(HZB_SPHERE, (0.7,)), (HZB_SPHEROID, (1.0, 1.3)), (HZB_SPHEROID, (1.0, 1.7))][q % 3]
            cen = np.array([5.0 * (q - 1), 0.2 * q, -0.1 * q])
            panels, modes = max(4, panels - 2 * (q % 3)), modes - 4 * (q % 3)
        out.append((kind, par, panels, c["gl"], modes, cen, turn))
    return out


def sizes_of(c):
    """[(rings, modes, shape)] of every body; bodies of one shape share their matrices."""
    return [(b[2] * b[3], b[4], (b[0], b[1], b[2], b[3], b[4])) for b in bodies_of(c)]


def directions(n, seed):
    g = np.random.default_rng(seed).standard_normal((n, 3))
    return g / np.linalg.norm(g, axis=1, keepdims=True)


# ------------------------------------------------------------------ one case

def solver_of(c, **options):
    s = Solver(c["k"], c["k"], Options(**options))
    for b in bodies_of(c):
        s.add_body(*b)
    if c["op"] != "sum":
        s.build_scattering_matrices()
    return s


def vectors(n, rhs, seed):
    """Krylov vectors: complex, of unit variance, in no particular order."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn((n, rhs), dtype=torch.complex128, device="cuda", generator=g)


def prepare(c, seed):
    op = c["op"]
    if op == "solve":
        s = solver_of(c, precision=HZB_PREC_FP64 if c["prec"] == "f64" else HZB_PREC_MIXED_FP32,
                      residual=HZB_PREC_DOUBLE_FLOAT)
        if c["eps"] > 0:
            s.compress(c["eps"])
        return {"case": c, "solver": s, "dirs": directions(c["rhs"], seed),
                "out": torch.empty((s.N, c["rhs"]), dtype=torch.complex128, device="cuda")}
    if op == "far":
        s = solver_of(c, precision=HZB_PREC_FP64, gmres_tol=1e-12)
        s.solve_plane_waves(directions(c["rhs"], seed))
        return {"case": c, "solver": s, "xhat": directions(c["points"], seed + 1)}
    s = solver_of(c)
    return {"case": c, "solver": s, "x": vectors(s.N, c["rhs"], seed)}


def run(state):
    c, s = state["case"], state["solver"]
    if c["op"] == "solve":
        s.solve_plane_waves(state["dirs"])
        return s.get_density(state["out"])
    if c["op"] == "far":
        return s.far_field(state["xhat"])
    call = {"sum": s.interbody, "dinv": s.local_inverse, "apply": s.apply}[c["op"]]
    y = call(state["x"], precision=PREC[c["prec"]])
    return y.to(torch.complex64) if c["prec"] == "f32" else y


def work(c):
    size, rhs = sizes_of(c), c["rhs"]
    n = [a * b for a, b, _ in size]
    total = sum(n)
    word = 8 if c["prec"] in ("f32", "mixed") else 16
    # B: 28 operations of the pair kernel and 8 for each right-hand side, per ordered pair
    pairs = float(total) ** 2 - sum(float(x) ** 2 for x in n)
    sums = pairs * (28 + 8 * rhs)
    # D^{-1}: two azimuthal FFTs and one complex matrix product per mode
    inverse = sum(8.0 * a * a * b * rhs + 10.0 * a * b * math.log2(b) * rhs for a, b, _ in size)
    blocks = word * sum(a * a * (b + 1) / 2 for a, b in {(a, b) for a, b, _ in size})
    node, vec = 56.0 * total, 16.0 * total * rhs
    if c["op"] == "sum":
        return {"bytes": node + 2 * vec, "flops": sums}
    if c["op"] == "dinv":
        return {"bytes": blocks + 2 * vec, "flops": inverse}
    if c["op"] == "apply":
        return {"bytes": node + blocks + 2 * vec, "flops": sums + inverse}
    if c["op"] == "far":
        return {"bytes": node + vec + 16.0 * c["points"] * rhs, "flops": c["points"] * float(total) * (20 + 8 * rhs)}
    # a mixed solve: about ten inner applies and two residuals (the accelerated one's are on
    # the skeletons, of about a third of the nodes)
    less = 0.1 if c["eps"] > 0 else 1.0
    return {"bytes": 12 * (node + blocks + 2 * vec), "flops": 12 * less * (sums + inverse)}


# ------------------------------------------------------------------ the same in 64 bits

def exact_sum(xyz, nrm, w, sizes, k, x):
    """B x by plain torch, each pair of nodes on different bodies once for both directions."""
    y = torch.zeros_like(x)
    off = np.concatenate([[0], np.cumsum(sizes)])
    ws = x * (w / (4.0 * math.pi))[:, None]

    def real_mm(gr, gi, v):
        a, b = gr @ v.real, gi @ v.imag
        return torch.complex(a - b, gr @ v.imag + gi @ v.real)

    for p in range(len(sizes)):
        for q in range(p + 1, len(sizes)):
            J = slice(int(off[q]), int(off[q + 1]))
            step = max(16, int(8e6 / sizes[q]))
            for i0 in range(int(off[p]), int(off[p + 1]), step):
                I = slice(i0, min(i0 + step, int(off[p + 1])))
                d = [xyz[I, a, None] - xyz[None, J, a] for a in range(3)]
                ir = (d[0] * d[0] + d[1] * d[1] + d[2] * d[2]).rsqrt_()
                kr = k / ir
                c, s = torch.cos(kr), torch.sin(kr)
                for side in (0, 1):
                    nn = nrm[J].T[:, None, :] if side == 0 else -nrm[I].T[:, :, None]
                    X = (nn[0] * d[0] + nn[1] * d[1] + nn[2] * d[2]) * ir * ir
                    A, B = X * ir, k * X + k * ir
                    gr, gi = c * A + s * B, s * A - c * B
                    if side == 0:
                        y[I] += real_mm(gr, gi, ws[J])
                    else:
                        y[J] += real_mm(gr.T, gi.T, ws[I])
    return y


def exact_inverse(s, c, x):
    """D^{-1} x from the scattering matrices: FFT, one product per mode, inverse FFT."""
    out, at, kept = torch.empty_like(x), 0, {}
    for b, (rings, modes, shape) in enumerate(sizes_of(c)):
        if shape not in kept:
            kept[shape] = torch.tensor(np.stack([s.get_modal_block(b, p, 1, rings) for p in range((modes + 1) // 2)]),
                                       device="cuda")
        S = kept[shape]
        n = rings * modes
        f = torch.fft.fft(x[at:at + n].reshape(rings, modes, -1), dim=1)
        p = [min(m, modes - m) for m in range(modes)]
        g = torch.stack([S[p[m]] @ f[:, m] for m in range(modes)], dim=1)
        out[at:at + n] = torch.fft.ifft(g, dim=1).reshape(n, -1)
        at += n
    return out


def exact(c, seed):
    if c["op"] == "solve":
        return None
    state = prepare(c, seed)
    s = state["solver"]
    xyz, nrm, w = (torch.tensor(a, device="cuda") for a in s.get_nodes())
    if c["op"] == "far":
        sig = torch.tensor(s.get_density(), device="cuda")
        xh = torch.tensor(state["xhat"], device="cuda")
        ph = torch.polar(torch.ones(1, dtype=torch.float64, device="cuda"), -c["k"] * (xh @ xyz.T))
        return ((ph * (-1j * (c["k"] * (xh @ nrm.T) + c["k"]))) @ (sig * (w / (4.0 * math.pi))[:, None])).cpu().numpy()
    sizes = [a * b for a, b, _ in sizes_of(c)]
    x = state["x"]
    if c["op"] == "sum":
        return exact_sum(xyz, nrm, w, sizes, c["k"], x)
    if c["op"] == "dinv":
        return exact_inverse(s, c, x)
    return x + exact_inverse(s, c, exact_sum(xyz, nrm, w, sizes, c["k"], x))
