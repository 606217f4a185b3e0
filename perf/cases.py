"""What a user of the library has it do, as measurable cases.

A case names one operation on one boundary integral system:

* ``assemble``     bm_assemble and the assembled blocks (a frequency sweep assembles anew per wavenumber);
* ``factor_solve`` bm_factor and bm_solve of an assembled system (the library's headline measure);
* ``solve``        bm_solve with kept factors (more incident waves on the same scatterer);
* ``far_field``    bm_far_field of given solutions;
* ``scatter``      the whole chain: assembly, plane-wave right-hand sides, factorisation, solve, far field;
* ``ssm``          the contour eigenvalue solver bm_ssm;
* ``serve``        a burst of requests through the serving loop bm_server_*.

The mixed-precision solves are refined to a backward error of 1e-14 with every residual formed afresh,
which is what a forward relative error of 1e-9 takes over this range: the default tolerance of 1e-9
bounds the residual only (forward errors reach 6e-9), updated residuals leave forward errors up to
5e-9, and a backward error of 1e-12 still left 3e-9 at 5700 nodes.  The seed draws the frequency (the
case's wavenumbers within 3 %), the incidence angles and the Gaussian data.
"""
import math

import numpy as np
import torch

from paper_2512_14193_gb300 import bm

CURVES = {  # kind, parameters (x(t) as in include/bm.h), rough diameter
    "circle": (bm.BM_CURVE_CIRCLE, (1.0, 0.0, 0.0, 0.0)),
    "ellipse": (bm.BM_CURVE_ELLIPSE, (1.0, 0.6, 0.0, 0.0)),
    "star": (bm.BM_CURVE_STAR, (1.0, 0.3, 5.0, 0.0)),
    "kite": (bm.BM_CURVE_KITE, (0.65, 1.5, 0.0, 0.0)),
}
PRECS = {"fp64": bm.BM_FP64, "tf32": bm.BM_CF32_TF32_IR, "3xtf32": bm.BM_CF32_3XTF32_IR}
TOL = 1e-14


def _case(op, curve, n, form, prec, k, kim=0.0, ratio=1.5, nrhs=1, angles=0, zeta_p=0, **more):
    return dict(op=op, curve=curve, n=n, form=form, prec=prec, k=k, kim=kim, ratio=ratio, nrhs=nrhs, angles=angles,
                zeta_p=zeta_p, **more)


def listed():
    return [
        # the smallest scatterer of the paper's section 5.1, in FP64, from curve to far field: launches and latency
        dict(_case("scatter", "circle", 256, "mixed", "fp64", 2.0, nrhs=1, angles=64), name="scatter circle 256 fp64"),
        # a lossy medium (complex wavenumber), a node count that fits no tile, the order-31 quadrature, the
        # ordinary formulation: the general call
        dict(_case("scatter", "star", 777, "ordinary", "3xtf32", 10.0, kim=-0.2, nrhs=17, angles=100, zeta_p=14),
             name="scatter star 777 lossy"),
        # one frequency of a sweep with a few incidence angles, from curve to far field
        dict(_case("scatter", "ellipse", 2048, "mixed", "3xtf32", 15.0, nrhs=8, angles=256), name="scatter ellipse 2048"),
        # assembly of the benchmark's operator
        dict(_case("assemble", "star", 4096, "mixed", "3xtf32", 20.0), name="assemble star 4096"),
        # the benchmark: factor + solve, 65 right-hand sides, mixed and ordinary formulation
        dict(_case("factor_solve", "star", 4096, "mixed", "3xtf32", 20.0, nrhs=65), name="factor solve star 4096"),
        dict(_case("factor_solve", "star", 4096, "ordinary", "3xtf32", 20.0, nrhs=65), name="factor solve ordinary 4096"),
        # the cheaper single-TF32 factors on a medium system
        dict(_case("factor_solve", "star", 1024, "mixed", "tf32", 8.0, nrhs=16), name="factor solve star 1024 tf32"),
        # FP64 throughout: the accuracy reference users compare with
        dict(_case("factor_solve", "kite", 1000, "mixed", "fp64", 10.0, nrhs=4), name="factor solve kite 1000 fp64"),
        # the large kite
        dict(_case("factor_solve", "kite", 8192, "mixed", "3xtf32", 50.0, nrhs=8), name="factor solve kite 8192"),
        # further incident waves on kept factors
        dict(_case("solve", "star", 4096, "mixed", "3xtf32", 20.0, nrhs=32), name="solve star 4096"),
        # the contour eigenvalue solver on the contour-batch workload's ellipse, around three resonances
        dict(_case("ssm", "ellipse", 1024, "mixed", "3xtf32", 5.2, kim=-1.05, nrhs=16, radius=0.3, points=32),
             name="ssm ellipse 1024"),
        # a burst of the serving stream
        dict(_case("serve", "star", 2048, "mixed", "3xtf32", 2.0, nrhs=64, requests=24), name="serve 24 requests"),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    op = rng.choices(["factor_solve", "scatter", "assemble", "solve", "far_field", "ssm", "serve"],
                     [35, 25, 12, 10, 8, 5, 5])[0]
    if op == "ssm":
        return _case(op, "ellipse", int(_log(rng, 200, 1024)), rng.choice(["mixed", "ordinary"]), "3xtf32", 5.2,
                     kim=-1.05, nrhs=rng.randint(4, 16), radius=0.3, points=rng.choice([16, 24, 32]))
    if op == "serve":
        return _case(op, "star", rng.choice([512, 1024, 2048]), "mixed", "3xtf32", 2.0, nrhs=rng.randint(8, 64),
                     requests=rng.randint(8, 24))
    form = rng.choice(["mixed", "mixed", "ordinary"])
    prec = rng.choices(["3xtf32", "tf32", "fp64"], [60, 15, 25])[0]
    top = {"3xtf32": 6000 if form == "mixed" else 4096, "tf32": 2048, "fp64": 1024}[prec]
    n = int(_log(rng, 200, top))
    # at least about twelve nodes per interior wavelength along the curve
    k = _log(rng, 2.0, max(2.5, min(40.0, n / 30.0)))
    kim = rng.choice([0.0, 0.0, -0.02 * k])
    return _case(op, rng.choice(sorted(CURVES)), n, form, prec, k, kim=kim, nrhs=int(_log(rng, 1, 65.99)),
                 angles=int(_log(rng, 16, 512)) if op in ("scatter", "far_field") else 0,
                 zeta_p=rng.choice([0, 0, 0, 14]) if op in ("scatter", "assemble") else 0)


class _Handle:
    """A library handle that goes with its state."""

    def __init__(self):
        self.h = bm.bm_create(0)

    def __del__(self):
        try:
            bm.bm_destroy(self.h)
        except Exception:  # the interpreter is shutting down
            pass


class _Server:
    def __init__(self, opts):
        self.s = bm.bm_server_create(0, slots=8, opts=opts)

    def __del__(self):
        try:
            bm.bm_server_destroy(self.s)
        except Exception:  # the interpreter is shutting down
            pass


def _rows(case):
    return (3 if case["form"] == "mixed" else 2) * case["n"]


def _form(case):
    return bm.BM_MIXED if case["form"] == "mixed" else bm.BM_ORDINARY


def _opts(case):
    return bm.make_opts(PRECS[case["prec"]], refine_tol=TOL, residual=bm.BM_RESID_TC_ALL, zeta_p=case["zeta_p"])


def _wavenumbers(case, rng):
    k = complex(case["k"], case["kim"]) * rng.uniform(0.97, 1.03)
    return k, case["ratio"] * k


def _gauss(rng, rows, cols):
    return np.asfortranarray((rng.normal(size=(cols, rows)) + 1j * rng.normal(size=(cols, rows))).T * math.sqrt(0.5))


def _device(a):
    """Column-major complex128 CUDA copy of a."""
    return torch.from_numpy(np.ascontiguousarray(a.T)).cuda().t()


def _empty(rows, cols):
    return torch.zeros((cols, rows), dtype=torch.complex128, device="cuda").t()


def _data(case, rng, k):
    """Right-hand sides of a factor_solve or solve: one plane wave, the rest Gaussian data on the curve."""
    n, rows = case["n"], _rows(case)
    b = np.zeros((rows, case["nrhs"]), dtype=np.complex128, order="F")
    off = 2 * n if case["form"] == "mixed" else 0
    b[off:off + n] = _gauss(rng, n, case["nrhs"])
    g = _geometry(case["curve"], n)
    a = rng.uniform(0.0, 2.0 * math.pi)
    b[off:off + n, 0] = _plane_wave(g, k, 1j / k, a)
    return b


def prepare(case, seed):
    rng = np.random.Generator(np.random.PCG64(int(seed)))
    op, n, rows = case["op"], case["n"], _rows(case)
    if op == "ssm":
        v = _gauss(rng, rows, case["nrhs"])
        center = complex(case["k"], case["kim"]) + 0.01 * complex(rng.uniform(-1, 1), rng.uniform(-1, 1))
        opts = bm.make_opts(PRECS[case["prec"]], refine_tol=1e-15, residual=bm.BM_RESID_TC_ALL)
        return dict(case=case, v=v, center=center, opts=opts)
    if op == "serve":
        return dict(case=case, server=_Server(_opts(case)), requests=_requests(case, rng))
    k0, k1 = _wavenumbers(case, rng)
    st = dict(case=case, k=(k0, k1), hold=_Handle(), opts=_opts(case))
    h = st["hold"].h
    kind, p = CURVES[case["curve"]]
    if op == "assemble":
        m, nb = (n, 4) if case["form"] == "mixed" else (2 * n, 1)
        st["out"] = [_empty(m, m) for _ in range(nb)]
        return st
    if op == "scatter":
        # the way a script uses the library: host angles in, host arrays out
        st["incident"] = rng.uniform(0.0, 2.0 * math.pi, case["nrhs"])
        st["observed"] = np.sort(rng.uniform(0.0, 2.0 * math.pi, case["angles"]))
        st["b"] = np.zeros((rows, case["nrhs"]), dtype=np.complex128, order="F")
        st["x"] = np.zeros((rows, case["nrhs"]), dtype=np.complex128, order="F")
        st["u"] = np.zeros((case["angles"], case["nrhs"]), dtype=np.complex128, order="F")
        return st
    bm.bm_assemble(h, kind, p, n, k0, k1, _form(case), st["opts"])
    if op == "far_field":
        st["observed"] = np.sort(rng.uniform(0.0, 2.0 * math.pi, case["angles"]))
        st["x"] = _device(_gauss(rng, rows, case["nrhs"]))
        st["u"] = _empty(case["angles"], case["nrhs"])
        return st
    st["b"] = _device(_data(case, rng, k0))
    st["x"] = _empty(rows, case["nrhs"])
    if op == "solve":
        bm.bm_factor(h)
    return st


def _requests(case, rng):
    """Requests with the serving stream's distributions, node counts up to the case's."""
    sizes = [v for v in (256, 512, 1024, 2048, 4096, 8192) if v <= case["n"]]
    out = []
    for i in range(case["requests"]):
        n = sizes[i % len(sizes)]  # each size equally often, so that every burst is the same amount of work
        nrhs = 1 + (i * 37) % case["nrhs"]
        k = complex(rng.uniform(2.0, min(40.0, n / 30.0)), rng.uniform(-0.5, 0.0))
        curve = (1.0, float(rng.uniform(0.1, 0.3)), float(rng.integers(3, 9)), 0.0)
        b = np.zeros((3 * n, nrhs), dtype=np.complex128, order="F")
        b[2 * n:] = _gauss(rng, n, nrhs)
        out.append((curve, n, k, b, np.zeros_like(b, order="F")))
    return out


def run(state):
    case = state["case"]
    op, n = case["op"], case["n"]
    kind, p = CURVES[case["curve"]]
    if op == "ssm":
        om, sigma, _ = bm.bm_ssm(0, kind, p, n, _form(case), state["opts"], state["center"], case["radius"],
                                 case["points"], 4, case["ratio"], state["v"], rank_tol=1e-2)
        return {"omega": om, "sigma": sigma}
    if op == "serve":
        s = state["server"].s
        tickets = [bm.bm_server_submit(s, bm.BM_CURVE_STAR, c, m, k, case["ratio"] * k, bm.BM_MIXED, b, x)
                   for c, m, k, b, x in state["requests"]]
        for t in tickets:
            r = bm.bm_server_wait(s, t)
            if r.status != bm.BM_OK:
                raise RuntimeError(f"request: {bm.bm_strerror(r.status)}")
        return [x for _, _, _, _, x in state["requests"]]
    h = state["hold"].h
    if op == "assemble":
        bm.bm_assemble(h, kind, p, n, *state["k"], _form(case), state["opts"])
        for q, t in enumerate(state["out"]):
            bm.bm_copy_block(h, q, t)
        return state["out"]
    if op == "scatter":
        bm.bm_assemble(h, kind, p, n, *state["k"], _form(case), state["opts"])
        bm.bm_rhs_plane_wave(h, state["incident"], state["b"])
        bm.bm_factor(h)
        bm.bm_solve(h, state["b"], state["x"])
        bm.bm_far_field(h, state["x"], state["observed"], state["u"])
        return {"x": state["x"], "u": state["u"]}
    if op == "far_field":
        bm.bm_far_field(h, state["x"], state["observed"], state["u"])
        return state["u"]
    if op == "factor_solve":
        bm.bm_factor(h)
    bm.bm_solve(h, state["b"], state["x"])
    return state["x"]


def _parts(op, form, n, prec, nrhs, angles):
    """(bytes, flops) of assembly, factorisation, solve and far field of one system."""
    mixed = form == "mixed"
    word = 16 if prec == "fp64" else 8  # of a stored factor
    rows, order = (3 * n, n) if mixed else (2 * n, 2 * n)
    by = fl = 0.0
    if op in ("assemble", "scatter"):
        by += 64.0 * n * n  # the four blocks written
        fl += 200.0 * n * n  # two Hankel pairs for each unordered pair of nodes
    if op in ("factor_solve", "scatter"):
        by += 64.0 * n * n + word * order * order
        fl += 8.0 / 3.0 * order ** 3 + (16.0 * n ** 3 if mixed else 0.0)
    if op in ("factor_solve", "solve", "scatter"):
        by += word * order * order + (4.0 * word * n * n if mixed else 0.0) + 32.0 * rows * nrhs
        fl += 8.0 * nrhs * (order * order + (4.0 * n * n if mixed else 0.0))
    if op in ("far_field", "scatter"):
        by += 16.0 * (2 * n * nrhs + angles * nrhs) + 56.0 * n
        fl += 16.0 * angles * n * nrhs + 60.0 * angles * n
    return by, fl


def work(case):
    if case["op"] == "ssm":
        got = [_parts("scatter", case["form"], case["n"], case["prec"], case["nrhs"], 0)] * case["points"]
    elif case["op"] == "serve":
        rng = np.random.Generator(np.random.PCG64(0))
        got = [_parts("scatter", "mixed", n, case["prec"], b.shape[1], 0) for _, n, _, b, _ in _requests(case, rng)]
    else:
        got = [_parts(case["op"], case["form"], case["n"], case["prec"], case["nrhs"], case["angles"])]
    return {"bytes": sum(g[0] for g in got), "flops": sum(g[1] for g in got)}


# ---- the same in 64 bits, plainly (the one-point rule) ----

def _geometry(curve, n):
    """x, y, nu_x, nu_y, |x'|, curvature, w at the n nodes."""
    t = 2.0 * math.pi * np.arange(n) / n
    s, c = np.sin(t), np.cos(t)
    p = CURVES[curve][1]
    if curve == "circle":
        x, y, dx, dy, ddx, ddy = p[0] * c, p[0] * s, -p[0] * s, p[0] * c, -p[0] * c, -p[0] * s
    elif curve == "ellipse":
        x, y, dx, dy, ddx, ddy = p[0] * c, p[1] * s, -p[0] * s, p[1] * c, -p[0] * c, -p[1] * s
    elif curve == "star":
        return _star(n, *p[:3])
    else:
        s2, c2 = np.sin(2 * t), np.cos(2 * t)
        x, y, dx, dy = c + p[0] * c2 - p[0], p[1] * s, -s - 2 * p[0] * s2, p[1] * c
        ddx, ddy = -c - 4 * p[0] * c2, -p[1] * s
    return _nodes(x, y, dx, dy, ddx, ddy)


def _star(n, r0, amp, lobes):
    t = 2.0 * math.pi * np.arange(n) / n
    s, c = np.sin(t), np.cos(t)
    r, dr = r0 + amp * np.cos(lobes * t), -amp * lobes * np.sin(lobes * t)
    ddr = -amp * lobes ** 2 * np.cos(lobes * t)
    return _nodes(r * c, r * s, dr * c - r * s, dr * s + r * c, ddr * c - 2 * dr * s - r * c,
                  ddr * s + 2 * dr * c - r * s)


def _nodes(x, y, dx, dy, ddx, ddy):
    sp = np.hypot(dx, dy)
    return x, y, dy / sp, -dx / sp, sp, (dx * ddy - dy * ddx) / sp ** 3, 2.0 * math.pi / x.size * sp


def _plane_wave(g, k, beta, a):
    ca, sa = math.cos(a), math.sin(a)
    u = np.exp(1j * k * (ca * g[0] + sa * g[1]))
    return -u * (1.0 + beta * 1j * k * (ca * g[2] + sa * g[3]))


def _hankel(z):
    """H0^(1), H1^(1) at complex z, Im z <= 0: J_m by backward recurrence (Miller), normalised by
    J0 + 2 (J2 + J4 + ...) = 1, Y0 by Neumann's series in J_2m, Y1 = -Y0'."""
    top = float(z.abs().max())
    m = 2 * int(0.5 * (top + 12.0 * top ** (1 / 3) + 30.0))
    hi, lo = torch.zeros_like(z), torch.full_like(z, 1e-30)  # J_{m+1}, J_m up to a factor
    norm, y0, y1 = torch.zeros_like(z), torch.zeros_like(z), torch.zeros_like(z)
    inv = 2.0 / z
    for j in range(m, 0, -1):  # lo is J_j
        q = j // 2
        if j % 2 == 0:
            norm += 2.0 * lo
            y0 += (-1.0) ** q / q * lo
        elif q > 0:
            y1 += (-1.0) ** q * (2 * q + 1) / (q * (q + 1)) * lo
        hi, lo = lo, j * inv * lo - hi
        if j % 4 == 0:  # keep the unnormalised values in range (small |z| grows fast)
            s = torch.where(lo.abs() > 1e40, torch.full_like(lo.real, 1e-60), torch.ones_like(lo.real))
            for v in (hi, lo, norm, y0, y1):
                v *= s
    norm += lo
    j0, j1 = lo / norm, hi / norm
    lg = torch.log(0.5 * z) + np.euler_gamma
    b0 = 2.0 / math.pi * lg * j0 - 4.0 / math.pi * y0 / norm
    b1 = -inv / math.pi * j0 + 2.0 / math.pi * ((lg - 1.0) * j1 - y1 / norm)
    return j0 + 1j * b0, j1 + 1j * b1


def _operators(g, k, dev):
    """S, D, D*, N of the one-point zeta-corrected rule at the wavenumber k."""
    n = g[0].size
    h = 2.0 * math.pi / n
    x, y, nx, ny, sp, ka, w = (torch.from_numpy(np.ascontiguousarray(v)).to(dev) for v in g)
    S, D, Ds, Nn = (torch.empty((n, n), dtype=torch.complex128, device=dev) for _ in range(4))
    for a in range(0, n, 512):  # rows a .. e at a time
        e = min(n, a + 512)
        dx, dy = x[a:e, None] - x[None, :], y[a:e, None] - y[None, :]
        r = torch.hypot(dx, dy)
        i = torch.arange(a, e, device=dev)
        r[i - a, i] = 1.0
        h0, h1 = _hankel(k * r.to(S.dtype))
        dni = dx * nx[a:e, None] + dy * ny[a:e, None]
        dnj = dx * nx[None, :] + dy * ny[None, :]
        nn = nx[a:e, None] * nx[None, :] + ny[a:e, None] * ny[None, :]
        pp = dni * dnj / (r * r)
        S[a:e] = 0.25j * h0 * w
        D[a:e] = 0.25j * k * h1 * (dnj / r) * w
        Ds[a:e] = -0.25j * k * h1 * (dni / r) * w
        Nn[a:e] = 0.25j * k * (k * h0 * pp + h1 * ((nn - 2.0 * pp) / r)) * w
    i = torch.arange(n, device=dev)
    S[i, i] = w * (0.25j - (np.log(complex(k) / 2.0) + np.euler_gamma) / (2 * math.pi)
                   - torch.log(w / (2 * math.pi)) / (2 * math.pi))
    D[i, i] = Ds[i, i] = (-ka * w / (4 * math.pi)).to(D.dtype)
    Nn[i, i] = -math.pi / (6.0 * h * sp) - k * k / (4 * math.pi) * math.log(h / (2 * math.pi)) * w.to(D.dtype)
    return S, D, Ds, Nn


def _blocks(case, k0, k1, dev, g=None):
    g = _geometry(case["curve"], case["n"]) if g is None else g
    eps1, beta = (k1 / k0) ** 2, 1j / k0
    S0, D0, Ds0, N0 = _operators(g, k0, dev)
    half = 0.5 * torch.eye(case["n"], dtype=torch.complex128, device=dev)
    m31 = D0 - half + beta * N0
    m32 = -(S0 + beta * (Ds0 + half))
    del S0, D0, Ds0, N0
    S1, D1, Ds1, _ = _operators(g, k1, dev)
    if case["form"] == "mixed":
        return [-S1, -(Ds1 + half) / eps1, m31, m32]
    return [torch.cat([torch.cat([m31, m32], 1), torch.cat([D1 + half, -eps1 * S1], 1)], 0)]


def _solution(case, blocks, b):
    if case["form"] != "mixed":
        return torch.linalg.solve(blocks[0], b)
    n = case["n"]
    m13, m23, m31, m32 = blocks
    x3 = torch.linalg.solve(-(m31 @ m13) - m32 @ m23, b[2 * n:] - m31 @ b[:n] - m32 @ b[n:2 * n])
    return torch.cat([b[:n] - m13 @ x3, b[n:2 * n] - m23 @ x3, x3], 0)


def _far(case, k, x, angles):
    g = _geometry(case["curve"], case["n"])
    n, ca, sa = case["n"], np.cos(angles)[:, None], np.sin(angles)[:, None]
    ph = g[6] * np.exp(-1j * k * (ca * g[0] + sa * g[1]))
    pre = np.exp(0.25j * math.pi) / np.sqrt(8.0 * math.pi * k)
    au = torch.from_numpy(pre * -1j * k * (ca * g[2] + sa * g[3]) * ph).to(x.device)
    return au @ x[:n] + torch.from_numpy(-pre * ph).to(x.device) @ x[n:2 * n]


def _resonances(case, seed, dev):
    """The block Sakurai-Sugiura steps of include/bm.h."""
    rng = np.random.Generator(np.random.PCG64(int(seed)))
    v = torch.from_numpy(_gauss(rng, _rows(case), case["nrhs"])).to(dev)
    center = complex(case["k"], case["kim"]) + 0.01 * complex(rng.uniform(-1, 1), rng.uniform(-1, 1))
    zeta = np.exp(2j * math.pi * (np.arange(case["points"]) + 0.5) / case["points"])
    mu = np.zeros((8, case["nrhs"], case["nrhs"]), dtype=np.complex128)
    for z in zeta:
        k = center + case["radius"] * z
        p = (v.conj().T @ _solution(case, _blocks(case, k, case["ratio"] * k, dev), v)).cpu().numpy()
        mu += (case["radius"] * z / case["points"] * z ** np.arange(8))[:, None, None] * p
    hankel = [np.block([[mu[i + j + s] for j in range(4)] for i in range(4)]) for s in (0, 1)]
    w1, sigma, w2 = np.linalg.svd(hankel[0])
    r = int((sigma > 1e-2 * sigma[0]).sum())
    lam = np.linalg.eigvals(w1[:, :r].conj().T @ hankel[1] @ w2[:r].conj().T / sigma[:r])
    om = center + case["radius"] * np.array(sorted(lam, key=lambda t: (abs(t) >= 1.0, t.real)))
    return {"omega": om, "sigma": sigma}


def exact(case, seed):
    op, n = case["op"], case["n"]
    if case["zeta_p"] != 0 or n > 6000:
        return None
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    if op == "ssm":
        return _resonances(case, seed, dev)
    rng = np.random.Generator(np.random.PCG64(int(seed)))
    if op == "serve":
        out = []
        for (r0, amp, lobes, _), m, k, b, _ in _requests(case, rng):
            one = dict(case, n=m)
            g = _star(m, r0, amp, lobes)
            out.append(_solution(one, _blocks(one, k, case["ratio"] * k, dev, g), torch.from_numpy(b).to(dev)))
        return out
    k0, k1 = _wavenumbers(case, rng)
    if op == "far_field":
        angles = np.sort(rng.uniform(0.0, 2.0 * math.pi, case["angles"]))
        return _far(case, k0, torch.from_numpy(_gauss(rng, _rows(case), case["nrhs"])).to(dev), angles)
    blocks = _blocks(case, k0, k1, dev)
    if op == "assemble":
        return blocks
    if op == "scatter":
        g = _geometry(case["curve"], n)
        incident = rng.uniform(0.0, 2.0 * math.pi, case["nrhs"])
        observed = np.sort(rng.uniform(0.0, 2.0 * math.pi, case["angles"]))
        b = np.zeros((_rows(case), case["nrhs"]), dtype=np.complex128)
        off = 2 * n if case["form"] == "mixed" else 0
        b[off:off + n] = np.stack([_plane_wave(g, k0, 1j / k0, a) for a in incident], 1)
        x = _solution(case, blocks, torch.from_numpy(b).to(dev))
        return {"x": x, "u": _far(case, k0, x, observed)}
    return _solution(case, blocks, torch.from_numpy(_data(case, rng, k0)).to(dev))
