"""The work that users of this engine have it do, as timed cases.

A case is one of
  run    a whole solve as the server and the command-line user make it: the initial
         state goes to the device, some macro steps of the multirate scheme with the
         limiters, the state comes back (``Solver.set_state``, ``step``, ``get_state``)
  rhs    one right-hand side R(Q) on the device (``Solver.rhs``)
  batch  an ensemble of uneven scenarios: states in, ``Batch.step``, states back

over the three scenarios of the benchmark: a hump on a flat bed (no limiter), the
wet/dry dam break (positivity and TVB limiters with M = 0) and the beach (graded,
jittered mesh, multirate levels, both limiters). Meshes and initial states come from
the seed; sizes, orders, tiers and schemes from the case. States of the single-
precision tiers are returned in single precision.

``exact`` evaluates the same discretisation in 64 bits with plain torch and numpy: the
pre-balanced form (free surface eta = h + B, pressure g/2 eta (eta - 2 B)) of the
nodal DG scheme of arXiv:1403.1661, multirate Adams-Bashforth of order 3, the
positivity limiter (its Algorithm 3) and the TVB limiter (its Section 5.3).
"""
import math

import numpy as np
import torch

G = 9.81
PP, TVB = 1, 2
DEVICE = "cuda" if torch.cuda.is_available() else "cpu"
SCENARIO = {   # limiter mask, dry threshold h0, TVB constant M
    "hump": (0, 1e-5, 0.0),
    "dam": (PP | TVB, 1e-5, 0.0),
    "beach": (PP | TVB, 1e-3, 1e-3),
}


def _case(name, kind, scenario, nx, ny, N, tier, levels, steps, scheme="cubature", compensated=False, trim=0,
          count=1):
    c = {"kind": kind, "scenario": scenario, "nx": nx, "ny": ny, "N": N, "tier": tier, "levels": levels,
         "steps": steps, "scheme": scheme, "compensated": compensated, "trim": trim, "count": count}
    return {"name": name, **c} if name else c


def listed():
    return [
        # the plain method on the smallest configured mesh, in double: launches and the
        # latency of one element's work
        _case("hump_512_n2_fp64", "run", "hump", 16, 16, 2, "fp64", 1, 100),
        # the wet/dry dam break at its configured size, limiters at every step
        _case("dam_20k_n3_fp32", "run", "dam", 320, 32, 3, "fp32", 1, 25),
        # a small and a middle request of the served stream (2k to 1M triangles, N = 2 to 4)
        _case("request_2k_n2_tc", "run", "beach", 64, 16, 2, "fp32tc", 4, 6),
        _case("request_45k_n3_tc", "run", "beach", 301, 75, 3, "fp32tc", 4, 25, trim=1),
        # the headline: the 500,000-triangle beach at N = 4, 200 finest substeps
        _case("beach_500k_n4_tc", "run", "beach", 1000, 250, 4, "fp32tc", 4, 25),
        # the same end to end, a snapshot after every macro step: transfers and one step
        _case("snapshot_500k_n4_tc", "run", "beach", 1000, 250, 4, "fp32tc", 4, 1),
        # one right-hand side: the headline mesh, and an odd size at the highest order
        # on the plain single-precision tier
        _case("rhs_500k_n4_tc", "rhs", "beach", 1000, 250, 4, "fp32tc", 4, 0),
        _case("rhs_75k_n5_fp32", "rhs", "beach", 387, 97, 5, "fp32", 4, 0, trim=1),
        # long runs that need the accuracy of double: the double tier, and the
        # compensated single-precision update
        _case("beach_40k_n4_fp64", "run", "beach", 283, 71, 4, "fp64", 4, 2, trim=1),
        _case("beach_100k_n3_comp", "run", "beach", 447, 112, 3, "fp32", 4, 10, compensated=True),
        # the cheaper collocation scheme
        _case("beach_125k_n4_colloc", "run", "beach", 500, 125, 4, "fp32tc", 4, 8, scheme="collocation"),
        # an ensemble of eight uneven scenarios, N = 3, 4, 5, advanced together
        _case("ensemble_8_tc", "batch", "beach", 5000, 100000, 0, "fp32tc", 4, 8, count=8),
    ]


def draw(rng):
    kind = rng.choice(["run", "run", "run", "run", "rhs", "rhs", "batch"])
    tier = rng.choice(["fp32tc", "fp32tc", "fp32tc", "fp32", "fp32", "fp64"])
    if kind == "batch":
        kmax = int(math.exp(rng.uniform(math.log(2e4), math.log(8e4))))
        return _case("", kind, "beach", rng.randint(2000, 6000), kmax, 0, rng.choice(["fp32tc", "fp32"]), 4,
                     rng.randint(1, 8), count=rng.randint(2, 8))
    scenario = rng.choice(["beach", "beach", "beach", "beach", "hump", "dam"])
    N = 3 if scenario == "dam" else rng.randint(2, 5)
    kmax = 2e5 if tier != "fp64" else 3e4
    K = math.exp(rng.uniform(math.log(1500.0 if scenario != "dam" else 8000.0), math.log(kmax)))
    if scenario == "hump":
        nx = ny = max(16, int(math.sqrt(K / 2)))
    else:
        ny = max(12, int(math.sqrt(K / (8 if scenario == "beach" else 20))))
        nx = int(K / (2 * ny))
    # runs stay within the time over which rounding does not grow: the thin layers of a
    # coarse shore, and of the dam's front, amplify it soon
    most = {"hump": 25, "dam": 25, "beach": 6 if K < 8e3 else 12 if K < 3e4 else 25}[scenario]
    work = 4e6 if tier != "fp64" else 8e4   # elements times macro steps
    steps = 0 if kind == "rhs" else max(1, min(rng.randint(3, most), int(work / (nx * ny * 2))))
    scheme = "cubature" if scenario == "dam" else rng.choice(["cubature"] * 6 + ["collocation", "cubature_2n"])
    if scheme == "collocation" and scenario == "beach" and kind == "run":
        scheme = "cubature"   # its aliasing is unstable at a coarse shore
    comp = tier != "fp64" and kind == "run" and rng.random() < 0.2
    return _case("", kind, scenario, nx, ny, N, tier, 4 if scenario == "beach" else 1, steps, scheme, comp,
                 rng.randint(0, 1))


# ---------------------------------------------------------------------------
# inputs


def _members(case):
    """The single-solver cases of an ensemble (sizes spread over their logarithm)."""
    if case["kind"] != "batch":
        return [case]
    out = []
    n = case["count"]
    for i in range(n):
        K = case["nx"] * (case["ny"] / case["nx"]) ** (((5 * i) % n) / max(n - 1, 1))
        ny = max(2, int(round(math.sqrt(K / 8.0))))
        out.append({**case, "nx": 4 * ny, "ny": ny, "N": 3 + i % 3})
    return out


def _mesh(case, rng):
    """Vertices and triangles: nx x ny cells cut in two, graded 8:1 and jittered on the beach."""
    nx, ny = case["nx"], case["ny"]
    x0, lx, ly = {"hump": (0.0, 1.0, 1.0), "dam": (0.0, 20.0, 2.0), "beach": (0.0, 400e3, 100e3)}[case["scenario"]]
    xs, ys = np.linspace(x0, lx, nx + 1), np.linspace(0.0, ly, ny + 1)
    if case["scenario"] == "beach":
        d = 0.125 ** (np.arange(nx) / max(nx - 1, 1))
        xs = np.concatenate([[0.0], np.cumsum(d)]) * (lx / d.sum())
    X, Y = (a.copy() for a in np.meshgrid(xs, ys))
    if case["scenario"] == "beach":
        d = np.diff(xs)
        X[:, 1:-1] += rng.uniform(-0.15, 0.15, (ny + 1, nx - 1)) * np.minimum(d[:-1], d[1:])
        Y[1:-1] += rng.uniform(-0.15, 0.15, (ny - 1, nx + 1)) * (ly / ny)
    v = np.arange((nx + 1) * (ny + 1)).reshape(ny + 1, nx + 1)
    a, b, c, d = v[:-1, :-1].ravel(), v[:-1, 1:].ravel(), v[1:, 1:].ravel(), v[1:, :-1].ravel()
    tri = np.stack([np.stack([a, b, c], 1), np.stack([a, c, d], 1)], 1).reshape(-1, 3).astype(np.int32)
    return X.ravel(), Y.ravel(), tri[:len(tri) - case["trim"]]


def _problem(case, seed):
    """The mesh, and the bed and initial depth as functions of (x, y, centroid x)."""
    rng = np.random.default_rng([seed, case["nx"], case["ny"], case["N"]])
    vx, vy, tri = _mesh(case, rng)
    if case["scenario"] == "hump":
        amp, cx, cy = rng.uniform(0.005, 0.02), rng.uniform(0.35, 0.65), rng.uniform(0.35, 0.65)
        bed = lambda x, y, c: np.full_like(x, -1.0)  # noqa: E731
        depth = lambda x, y, c, B: amp * np.exp(-((x - cx) ** 2 + (y - cy) ** 2) / 0.01) - B  # noqa: E731
    elif case["scenario"] == "dam":
        h, at = rng.uniform(0.8, 1.2), 20.0 * rng.integers(2 * case["nx"] // 5, 3 * case["nx"] // 5) / case["nx"]
        bed = lambda x, y, c: np.zeros_like(x)  # noqa: E731
        depth = lambda x, y, c, B: np.where(c < at, h, 0.0) + 0.0 * x  # noqa: E731
    else:
        amp, cx, cy = rng.uniform(0.5, 5.0), rng.uniform(20e3, 200e3), rng.uniform(10e3, 90e3)
        bed = lambda x, y, c: 2005.0 * (1.0 + np.tanh((x - 380e3) / 5e3)) - 4000.0  # noqa: E731
        depth = lambda x, y, c, B: np.maximum(  # noqa: E731
            0.0, amp * np.exp(-((x - cx) ** 2 + (y - cy) ** 2) / 1e8) - B)
    return vx, vy, tri, bed, depth


def _nodal(x, y, cx, bed, depth):
    B = bed(x, y, cx[:, None] + 0.0 * x)
    return B, depth(x, y, cx[:, None] + 0.0 * x, B)


def _momentum(case, x, y, h):
    """A current, so that both momenta carry values from the start: slow at sea, 1.5 m/s along
    and across the channel behind the dam."""
    if case["scenario"] == "dam":
        return 1.5 * h, 1.5 * h
    return 0.02 * h * np.sin(x / x.max() * 3.0), 0.01 * h * np.cos(y / y.max() * 2.0)


# ---------------------------------------------------------------------------
# the framework's part


def _solver(case, seed):
    import paper_1403_1661_gb300 as P

    vx, vy, tri, bed, depth = _problem(case, seed)
    mask, h0, M = SCENARIO[case["scenario"]]
    mesh = P.Mesh(vx, vy, tri)
    s = P.Solver(mesh, case["N"], g=G, h0=h0, cfl=0.5, nlevels_max=case["levels"], precision=case["tier"],
                 limiter_mask=mask, tvb_M=M, scheme=case["scheme"], compensated=case["compensated"])
    x, y = mesh.node_coords(case["N"])
    B, h = _nodal(x, y, mesh.centroids()[0], bed, depth)
    # page-locked host arrays for the state and its read-back, and the read-back in the
    # tier's own precision
    host = [torch.empty(h.shape, dtype=torch.float64, pin_memory=True) for _ in range(6)]
    init = [t.numpy() for t in host[:3]]
    init[0][:] = h
    init[1][:], init[2][:] = _momentum(case, x, y, h)
    s.set_bathymetry(B)
    s.set_state(*init)
    s.setup_levels()
    single = None if case["tier"] == "fp64" else [torch.empty(h.shape, dtype=torch.float32) for _ in range(3)]
    return {"solver": s, "init": init, "host": host[3:], "out": [t.numpy() for t in host[3:]], "single": single}


def prepare(case, seed):
    st = {"case": case, "members": [_solver(c, seed + 1000003 * i) for i, c in enumerate(_members(case))]}
    if case["kind"] == "batch":
        import paper_1403_1661_gb300 as P

        st["batch"] = P.Batch([m["solver"] for m in st["members"]], max_macro=max(1, case["steps"]))
    return st


def _read(m):
    m["solver"].get_state(out=m["out"])
    if m["single"] is None:
        return list(m["out"])
    for f, d in zip(m["single"], m["host"]):
        f.copy_(d)
    return list(m["single"])


def run(state):
    case, members = state["case"], state["members"]
    if case["kind"] == "rhs":
        return members[0]["solver"].rhs()
    for m in members:
        m["solver"].set_state(*m["init"])
    if case["kind"] == "batch":
        state["batch"].step(case["steps"])
    else:
        members[0]["solver"].step(case["steps"])
    return [_read(m) for m in members]


def work(case):
    """State, bed and history read and written once per element and stage (16 Np + 16 words,
    17 bytes), initial state and result crossing the bus once in 64 bits; the multiply-adds of
    the interpolations, projections and lifts."""
    total = {"bytes": 0.0, "flops": 0.0}
    for c in _members(case):
        N, s = c["N"], 8 if c["tier"] == "fp64" else 4
        K = 2 * c["nx"] * c["ny"] - c["trim"]
        np_, nc, ng = _sizes(N, c["scheme"])
        mads = 14 * np_ * nc + 9 * ng * np_ + 24 * ng * (N + 1) if c["scheme"] != "collocation" else (
            8 * np_ * np_ + 9 * ng * np_)
        if c["kind"] == "rhs":
            total["bytes"] += K * ((7 * np_ + 8) * s + 1)
            total["flops"] += 2.0 * K * mads
        else:
            # about 4.05 evaluations per element and macro step on the graded beach
            ev = c["steps"] * K * (4.05 if c["scenario"] == "beach" else 1.0)
            total["bytes"] += ev * ((16 * np_ + 16) * s + 17) + 6 * 8 * K * np_
            total["flops"] += 2.0 * ev * mads
    return total


def _sizes(N, scheme):
    np_ = (N + 1) * (N + 2) // 2
    if scheme == "collocation":
        return np_, np_, N + 1
    q = N + 1 if scheme == "cubature_2n" else (3 * N + 1) // 2
    return np_, q * q, N + 1 if scheme == "cubature_2n" else (3 * N + 2) // 2


# ---------------------------------------------------------------------------
# the same in 64 bits


def _gauss_jacobi10(q):
    """Gauss rule for the weight 1 - b on [-1, 1], by the eigenvalues of its Jacobi matrix."""
    k = np.arange(q)
    off = np.sqrt(k[1:] * (k[1:] + 1.0)) / (2.0 * k[1:] + 1.0)
    x, V = np.linalg.eigh(np.diag(-1.0 / ((2 * k + 1.0) * (2 * k + 3.0))) + np.diag(off, 1) + np.diag(off, -1))
    return x, 2.0 * V[0] ** 2


def _conical(q):
    """Points (r, s) and weights of the conical product rule on the reference triangle."""
    a, wa = np.polynomial.legendre.leggauss(q)
    b, wb = _gauss_jacobi10(q)
    A, Bb = np.meshgrid(a, b, indexing="ij")
    return ((1 + A) * (1 - Bb) / 2 - 1).ravel(), Bb.ravel(), (np.outer(wa, wb) / 2).ravel()


def _basis(N, r, s):
    """P_i(r) P_j(s), i + j <= N, and its derivatives."""
    leg = np.polynomial.legendre
    val, dr, ds = [], [], []
    for j in range(N + 1):
        for i in range(N + 1 - j):
            ci, cj = np.eye(N + 2)[i], np.eye(N + 2)[j]
            pi, pj = leg.legval(r, ci), leg.legval(s, cj)
            val.append(pi * pj)
            dr.append(leg.legval(r, leg.legder(ci)) * pj)
            ds.append(pi * leg.legval(s, leg.legder(cj)))
    return np.stack(val, 1), np.stack(dr, 1), np.stack(ds, 1)


def _nodes(N):
    """Warp & Blend nodes (Warburton 2006), row by row from the edge between vertices 0 and 1."""
    lam = np.array([[1 - (i + j) / N, i / N, j / N] for j in range(N + 1) for i in range(N + 1 - j)])
    alpha = {1: 0.0, 2: 0.0, 3: 1.4152, 4: 0.1001, 5: 0.2751}[N]
    inner = np.polynomial.legendre.Legendre.basis(N).deriv().roots() if N > 1 else np.zeros(0)
    gll, eq = np.concatenate([[-1.0], np.sort(np.real(inner)), [1.0]]), np.linspace(-1, 1, N + 1)

    def warp(x):
        out = np.zeros_like(x)
        for i in range(N + 1):
            p = np.ones_like(x)
            for j in range(N + 1):
                if j != i:
                    p *= (x - eq[j]) / (eq[i] - eq[j])
            out += (gll[i] - eq[i]) * p
        inside = np.abs(x) < 1 - 1e-10
        return np.where(inside, out / np.where(inside, 1 - x * x, 1.0), 0.0)

    v = np.array([[-1, -1 / math.sqrt(3)], [1, -1 / math.sqrt(3)], [0, 2 / math.sqrt(3)]])
    xy = lam @ v
    for a, b, c in ((0, 1, 2), (1, 2, 0), (2, 0, 1)):
        la, lb, lc = lam[:, a], lam[:, b], lam[:, c]
        # between the end points 1 - xi^2 = 4 la lb on the edge itself
        w = 4 * la * lb * warp(lb - la) * (1 + (alpha * lc) ** 2)
        xy = xy + w[:, None] * (v[b] - v[a]) / 2
    T = np.linalg.inv(np.vstack([v.T, np.ones(3)]))
    lam = np.hstack([xy, np.ones((len(xy), 1))]) @ T.T
    return lam


def _reference(N, scheme):
    lam = _nodes(N)
    r, s = 2 * lam[:, 1] - 1, 2 * lam[:, 2] - 1
    inv = np.linalg.inv(_basis(N, r, s)[0])
    at = lambda r, s: [b @ inv for b in _basis(N, r, s)]  # noqa: E731
    rc, sc, wc = _conical((3 * N + 1) // 2 if scheme != "cubature_2n" else N + 1)
    Ic, Icr, Ics = at(rc, sc)
    M = Ic.T @ (wc[:, None] * Ic)
    Mi = np.linalg.inv(M)
    proj = lambda A: Mi @ (A.T * wc)  # noqa: E731
    Pr, Ps, Pm = proj(Icr), proj(Ics), proj(Ic)
    lc = np.stack([-(rc + sc) / 2, (1 + rc) / 2, (1 + sc) / 2], 1)
    T1 = np.linalg.inv(lc.T @ (wc[:, None] * lc)) @ ((lc.T * wc) @ Ic)
    row = lambda j: j * (N + 1) - j * (j - 1) // 2  # noqa: E731
    face = np.array([[m for m in range(N + 1)], [row(m) + N - m for m in range(N + 1)],
                     [row(N - m) for m in range(N + 1)]])
    tg, wg = np.polynomial.legendre.leggauss((3 * N + 2) // 2 if scheme != "cubature_2n" else N + 1)
    ends = np.array([[-1.0, -1.0], [1.0, -1.0], [-1.0, 1.0]])
    I1d, Lg = None, []
    for f in range(3):
        p = np.outer((1 - tg) / 2, ends[f]) + np.outer((1 + tg) / 2, ends[(f + 1) % 3])
        E = at(p[:, 0], p[:, 1])[0]
        I1d = E[:, face[f]]
        Lg.append(Mi @ (E.T * wg))
    if scheme == "collocation":
        Dr, Ds = Pm @ Icr, Pm @ Ics
        Ic, Icr, Ics, Pr, Ps, Pm = np.eye(len(r)), Dr, Ds, Mi @ Dr.T @ M, Mi @ Ds.T @ M, np.eye(len(r))
        Lg, I1d = [L @ I1d for L in Lg], np.eye(N + 1)
    dev = lambda a: torch.as_tensor(np.ascontiguousarray(a), device=DEVICE)  # noqa: E731
    return {"lam": lam, "Ic": dev(Ic), "Icr": dev(Icr), "Ics": dev(Ics), "Pr": dev(Pr), "Ps": dev(Ps), "P": dev(Pm),
            "face": dev(face), "I1d": dev(I1d), "Lg": dev(np.concatenate(Lg, 1)), "mw": dev(wc @ Ic if scheme != "collocation" else M.sum(0)) / 2.0,
            "T1": dev(T1), "bary": dev(lam)}


def _geometry(vx, vy, tri):
    x, y = vx[tri], vy[tri]
    K = len(tri)
    xr, xs, yr, ys = (x[:, 1] - x[:, 0]) / 2, (x[:, 2] - x[:, 0]) / 2, (y[:, 1] - y[:, 0]) / 2, (y[:, 2] - y[:, 0]) / 2
    J = xr * ys - xs * yr
    rx, ry, sx, sy = ys / J, -xs / J, -yr / J, xr / J
    nxt = [1, 2, 0]
    a, b = tri, tri[:, nxt]
    key = (np.minimum(a, b).astype(np.int64) * len(vx) + np.maximum(a, b)).ravel()
    order = np.argsort(key, kind="stable")
    same = key[order][1:] == key[order][:-1]
    p, q = order[:-1][same], order[1:][same]
    other = np.full(3 * K, -1)
    other[p], other[q] = q, p
    vn = np.stack([np.stack([-sx, rx + sx, -rx], 1), np.stack([-sy, ry + sy, -ry], 1)])   # (sJ/J) n
    size = np.hypot(vn[0], vn[1])
    # TVB stencil: midpoint minus centroid as a combination of two neighbour centroids
    c = np.stack([x.mean(1), y.mean(1)])
    mid = np.stack([(x + x[:, nxt]) / 2, (y + y[:, nxt]) / 2]) - c[:, :, None]
    nb = other.reshape(K, 3)
    n = vn / size
    ghost = 2 * (mid * n).sum(0) * n
    db = np.where(nb >= 0, c[:, np.maximum(nb, 0) // 3] - c[:, :, None], ghost)
    best, alpha, beta, pick = np.full((K, 3), -np.inf), np.zeros((K, 3)), np.zeros((K, 3)), np.zeros((K, 3), int)
    for i in range(3):
        for j in ((i + 1) % 3, (i + 2) % 3):
            det = db[0, :, i] * db[1, :, j] - db[0, :, j] * db[1, :, i]
            al = (mid[0, :, i] * db[1, :, j] - db[0, :, j] * mid[1, :, i]) / det
            be = (db[0, :, i] * mid[1, :, i] - db[1, :, i] * mid[0, :, i]) / det
            up = np.minimum(al, be) > best[:, i]
            best[up, i], alpha[up, i], beta[up, i], pick[up, i] = np.minimum(al, be)[up], al[up], be[up], j
    dev = lambda a: torch.as_tensor(np.ascontiguousarray(a), device=DEVICE)  # noqa: E731
    length = np.hypot(x[:, nxt] - x, y[:, nxt] - y).sum(1)
    return {"rx": dev(rx)[:, None], "ry": dev(ry)[:, None], "sx": dev(sx)[:, None], "sy": dev(sy)[:, None],
            "other": dev(np.maximum(other, 0)).reshape(K, 3), "inner": dev(other >= 0).reshape(K, 3),
            "size": dev(size), "nx": dev(n[0]), "ny": dev(n[1]), "area": dev(2 * J), "H": dev(4 * J / length),
            "mid": dev(mid), "alpha": dev(alpha), "beta": dev(beta), "pick": dev(pick)}


class _Exact:
    def __init__(self, case, seed):
        vx, vy, tri, bed, depth = _problem(case, seed)
        self.case, self.ref, self.geo = case, _reference(case["N"], case["scheme"]), _geometry(vx, vy, tri)
        lam = self.ref["lam"]
        x, y = vx[tri] @ lam.T, vy[tri] @ lam.T
        B, h = _nodal(x, y, vx[tri].mean(1), bed, depth)
        hu, hv = _momentum(case, x, y, h)
        dev = lambda a: torch.as_tensor(a, device=DEVICE)  # noqa: E731
        self.B = dev(B)
        self.mask, self.h0, self.M = SCENARIO[case["scenario"]]
        self.hvel = self.h0 * (1 + 1e-6)
        o, g = self.ref, self.geo
        Br, Bs = self.B @ o["Icr"].T, self.B @ o["Ics"].T
        self.Bc = self.B @ o["Ic"].T
        self.Bx, self.By = g["rx"] * Br + g["sx"] * Bs, g["ry"] * Br + g["sy"] * Bs
        self.Bbar, self.Bv = self.B @ o["mw"], self.B @ o["T1"].T
        self.q = torch.stack([dev(h) + self.B, dev(hu), dev(hv)])
        K = len(tri)
        self.mean, self.dry = torch.zeros(3, K, dtype=torch.float64, device=DEVICE), torch.zeros(K, dtype=torch.bool, device=DEVICE)
        self.limit(self.q, torch.ones(K, dtype=torch.bool, device=DEVICE))

    def _faces(self, q):
        """Traces at the face points, own and across (walls mirrored)."""
        o, g = self.ref, self.geo
        own = q[:, :, o["face"]] @ o["I1d"].T                    # field, element, face, point
        far = own.reshape(len(q), -1, own.shape[-1])[:, g["other"]].flip(-1)
        inner = g["inner"][None, :, :, None]
        far = torch.where(inner, far, own)
        nx, ny = g["nx"][..., None], g["ny"][..., None]
        mn = own[1] * nx + own[2] * ny
        far[1], far[2] = far[1] - 2 * mn * nx * ~inner[0], far[2] - 2 * mn * ny * ~inner[0]
        return own, far, nx, ny

    def rhs(self, q):
        o, g, hv_ = self.ref, self.geo, self.hvel
        e, mu, mv = (q[f] @ o["Ic"].T for f in range(3))
        h = e - self.Bc
        inv = torch.where(h > hv_, 1 / h, torch.zeros_like(h))
        u, v, p = mu * inv, mv * inv, 0.5 * G * e * (h - self.Bc)
        a, b = g["rx"] * mu + g["ry"] * mv, g["sx"] * mu + g["sy"] * mv
        R = torch.stack([
            a @ o["Pr"].T + b @ o["Ps"].T,
            (u * a + g["rx"] * p) @ o["Pr"].T + (u * b + g["sx"] * p) @ o["Ps"].T - (G * e * self.Bx) @ o["P"].T,
            (v * a + g["ry"] * p) @ o["Pr"].T + (v * b + g["sy"] * p) @ o["Ps"].T - (G * e * self.By) @ o["P"].T])
        m, f, nx, ny = self._faces(torch.cat([q, self.B[None]]))
        hm, hp = m[0] - m[3], f[0] - f[3]
        zero = torch.zeros_like(hm)
        im, ip = torch.where(hm > hv_, 1 / hm, zero), torch.where(hp > hv_, 1 / hp, zero)
        um, vm, up, vp = m[1] * im, m[2] * im, f[1] * ip, f[2] * ip
        top = torch.maximum(m[3], f[3])
        sm, sp = (m[0] - top).clamp(min=0), (f[0] - top).clamp(min=0)
        cm, cp = um * nx + vm * ny, up * nx + vp * ny
        speed = torch.maximum(cm.abs() + (G * sm).sqrt(), cp.abs() + (G * sp).sqrt())
        pres = 0.5 * G * m[0] * (hm - m[3]) + 0.25 * G * (sp - sm) * (sp + sm)
        F = torch.stack([0.5 * (sm * cm + sp * cp - speed * (sp - sm)),
                         0.5 * (sm * cm * um + sp * cp * up - speed * (sp * up - sm * um)) + pres * nx,
                         0.5 * (sm * cm * vm + sp * cp * vp - speed * (sp * vp - sm * vm)) + pres * ny])
        F = F * g["size"][None, :, :, None]
        return R - F.reshape(3, F.shape[1], -1) @ o["Lg"].T

    def limit(self, q, act):
        """Positivity, then TVB, on the active elements of q, in place."""
        o = self.ref
        w = o["mw"]
        h = q[0] - self.B
        hb, ub, vb = h @ w, q[1] @ w, q[2] @ w
        dry = torch.zeros_like(act)
        if self.mask & PP:
            trig = h.amin(1) <= self.h0
            dry = trig & (hb < 1.01 * self.h0)
            h1 = h @ o["T1"].T
            den = hb - h1.amin(1)
            th = torch.where(den > 0, ((hb - self.h0) / den).clamp(max=1.0), torch.ones_like(den))[:, None]
            wet, off = (trig & ~dry & act)[:, None], (dry & act)[:, None]
            for f, (z, zb) in enumerate(((h, hb), (q[1], ub), (q[2], vb))):
                new = th * ((z @ o["T1"].T) @ o["bary"].T - zb[:, None]) + zb[:, None]
                q[f] = torch.where(wet, new + self.B if f == 0 else new, q[f])
                q[f] = torch.where(off, self.h0 + self.B if f == 0 else torch.zeros_like(q[f]), q[f])
            hb = torch.where(dry, torch.full_like(hb, self.h0), hb)
            ub, vb = torch.where(dry, 0 * ub, ub), torch.where(dry, 0 * vb, vb)
        self.mean = torch.where(act, torch.stack([hb + self.Bbar, ub, vb]), self.mean)
        self.dry = torch.where(act, dry, self.dry)
        if self.mask & TVB:
            self._tvb(q, act)

    def _tvb(self, q, act):
        o, g = self.ref, self.geo
        nb = g["other"] // 3
        near_dry = (self.dry[nb] & g["inner"]).any(1)
        e = torch.nonzero(act & ~self.dry & ~near_dry)[:, 0]
        u0 = self.mean[:, e]                                     # field, element
        un = torch.where(g["inner"][e], self.mean[:, nb[e]], u0[:, :, None])
        mn = u0[1][:, None] * g["nx"][e] + u0[2][:, None] * g["ny"][e]
        out = ~g["inner"][e]
        un[1], un[2] = un[1] - 2 * mn * g["nx"][e] * out, un[2] - 2 * mn * g["ny"][e] * out
        vq = q[:, e] @ o["T1"].T
        nxt = [1, 2, 0]
        dt = (vq + vq[..., nxt]) / 2 - u0[..., None]             # field, element, edge
        far = torch.gather(un, 2, g["pick"][e].expand(3, -1, -1))
        dn = g["alpha"][e] * (un - u0[..., None]) + g["beta"][e] * (far - u0[..., None])
        hb = u0[0] - self.Bbar[e]
        c, u, v = (G * hb).sqrt()[:, None], (u0[1] / hb)[:, None], (u0[2] / hb)[:, None]
        mid = g["mid"][:, e]
        dist = (mid ** 2).sum(0).sqrt()
        nx, ny = mid[0] / dist, mid[1] / dist

        def waves(d):   # left eigenvectors: fast -, shear, fast +
            un_, s = (d[1] - u * d[0]) * nx + (d[2] - v * d[0]) * ny, (d[2] - v * d[0]) * nx - (d[1] - u * d[0]) * ny
            return torch.stack([0.5 * (d[0] - un_ / c), s, 0.5 * (d[0] + un_ / c)])

        wt, wn = waves(dt), 1.5 * waves(dn)
        floor = 1e-6 * (hb + (u0[1] ** 2 + u0[2] ** 2).sqrt() / c[:, 0])
        thr = self.M * dist ** 2 + floor[:, None]
        thr = torch.stack([thr, thr * c, thr])
        mm = torch.where(wt.sign() * wn.sign() > 0, wt.sign() * torch.minimum(wt.abs(), wn.abs()), torch.zeros_like(wt))
        wl = torch.where(wt.abs() <= thr, wt, mm)
        hit = (wl != wt).any(0).any(1)
        d = torch.stack([wl[0] + wl[2], u * (wl[0] + wl[2]) + c * nx * (wl[2] - wl[0]) - ny * wl[1],
                         v * (wl[0] + wl[2]) + c * ny * (wl[2] - wl[0]) + nx * wl[1]])
        pos, neg = d.clamp(min=0).sum(2), (-d).clamp(min=0).sum(2)
        one = torch.ones_like(pos)
        tp = torch.where(pos > 0, (neg / pos).clamp(max=1.0), one)[..., None]
        tn = torch.where(neg > 0, (pos / neg).clamp(max=1.0), one)[..., None]
        d = tp * d.clamp(min=0) - tn * (-d).clamp(min=0)
        Bv = self.Bv[e]
        dh = d[0] - ((Bv + Bv[:, nxt]) / 2 - self.Bbar[e][:, None])
        vertex = lambda d: torch.stack([d[..., 0] + d[..., 2] - d[..., 1], d[..., 1] + d[..., 0] - d[..., 2],  # noqa: E731
                                        d[..., 2] + d[..., 1] - d[..., 0]], -1)
        low, avg = vertex(dh).amin(1), dh.mean(1)
        den = avg - low
        th = torch.where(den > 0, ((hb + avg - self.h0) / den).clamp(0.0, 1.0), torch.ones_like(den))
        th = torch.where(hb + low < self.h0, th, torch.ones_like(th))[:, None]
        dh = avg[:, None] + th * (dh - avg[:, None])
        k = e[hit]
        q[0, k] = (hb[hit][:, None] + vertex(dh[hit])) @ o["bary"].T + self.B[k]
        for f in (1, 2):
            q[f, k] = (u0[f][hit][:, None] + vertex(d[f][hit])) @ o["bary"].T

    def levels(self):
        h = self.q[0] - self.B
        ref = 1e-2 * h.max()
        safe = torch.where(h > ref, h, torch.full_like(h, math.inf))
        a = torch.hypot(self.q[1] / safe, self.q[2] / safe) + (G * h.clamp(min=ref)).sqrt()
        dt = 0.5 / (self.case["N"] + 1.0) ** 2 * self.geo["H"] / a.amax(1)
        lev = torch.frexp(dt / dt.min())[1].clamp(1, self.case["levels"])
        return lev, float(dt.min())

    def steps(self, n):
        """n macro steps of the multirate Adams-Bashforth scheme of order 3."""
        dev = lambda a: torch.as_tensor(a, device=DEVICE)  # noqa: E731
        lev, dtm = self.levels()
        L, dt = int(lev.max()), (dtm * 2.0 ** (lev - 1).double())[None, :, None]
        end, start = self.q, self.q.clone()
        hist = [torch.zeros_like(end) for _ in range(3)]
        for k in range(n * 2 ** (L - 1)):
            per = 2 ** (lev - 1).long()
            act, a = (k % per) == 0, torch.div(k, per, rounding_mode="floor")
            A = act[None, :, None]
            start = torch.where(A, end, start)
            view = start
            if L > 1:
                x, full, one = (k % per).double() / per, a >= 2, a == 1
                w = [torch.where(full, x ** 3 / 6 + 0.75 * x ** 2 + x, torch.where(one, x + 0.5 * x * x, x)),
                     torch.where(full, -(x ** 3 / 3 + x ** 2), torch.where(one, -0.5 * x * x, 0 * x)),
                     torch.where(full, x ** 3 / 6 + 0.25 * x ** 2, 0 * x)]
                view = start + dt * sum(w[s][None, :, None] * hist[s] for s in range(3))
            R = self.rhs(view)
            hist = [torch.where(A, new, old) for new, old in zip([R, hist[0], hist[1]], hist)]
            depth = a.clamp(max=2)
            ab = dev(np.array([[1, 0, 0], [1.5, -0.5, 0], [23 / 12, -16 / 12, 5 / 12]]))[depth]
            new = start + dt * sum(ab[:, s][None, :, None] * hist[s] for s in range(3))
            end = torch.where(A, new, end)
            self.limit(end, act)
        self.q = end


def exact(case, seed):
    out = []
    for i, c in enumerate(_members(case)):
        x = _Exact(c, seed + 1000003 * i)
        if case["kind"] == "rhs":
            return x.rhs(x.q)
        x.steps(case["steps"])
        out.append([x.q[0] - x.B, x.q[1], x.q[2]])
    return out
