"""The measured work of the multibody scattering library: single calls and whole solves.

A case names a body family (`geo`), its size and the call (`do`):
  geo "star"      the 10-body grid of 3-stars at kappa = 10 (mbs_inputs.config0);
  geo "lattice"   circles, 3-stars and ellipses sharing 3 shapes on a jittered lattice, 64 skeleton points each (config1);
  geo "sizes"     2D bodies of uneven size, each its own shape, 35 to 105 skeleton points (config2);
  geo "ellipsoids"  3D, each its own shape, 300 skeleton points (config3);
  geo "coarse3d"  3D ellipsoids on a coarse grid, each its own shape, 90 skeleton points (tiny_3d).
Vectors are (rows, right-hand sides) complex128 on the GPU, the layout that the binding takes without a copy.
"""
import math

import numpy as np
import torch

import mbs_inputs as mi
import paper_2603_19113_gb300 as mbs

DEV = "cuda"


# ---------------------------------------------------------------- the cases
def listed():
    return [
        # the smallest call: the README's sequence on ten bodies, everything in FP64 (the library's default), one plane wave;
        # launches and latency count
        dict(name="whole_10_fp64", do="whole", geo="star", T=10, kappa=10.0, nrhs=1, M=257, tol=1e-11),
        # the headline in small: mixed-precision solve for 8 plane waves at kappa = 40 (rhs, then FP32 block GMRES in FP64 refinement)
        dict(name="solve_160_mixed", do="solve", geo="lattice", T=160, kappa=40.0, nrhs=8, tol=1e-11),
        # set-up of a request: 3 shapes shared by 1000 bodies, so few shapes and long chains
        dict(name="build_3_shapes", do="build", geo="lattice", T=1000, kappa=40.0),
        # set-up where every body is its own shape: throughput
        dict(name="build_300_sizes", do="build", geo="sizes", T=300, kappa=20.0),
        # 3D set-up of a few shapes
        dict(name="build_6_coarse3d", do="build", geo="coarse3d", T=6, kappa=3.0),
        # right-hand sides of the 1000-body workload
        dict(name="rhs_1000", do="rhs", geo="lattice", T=1000, kappa=40.0, nrhs=8),
        # the operator of the Krylov steps in FP32: the 1000-body headline workload, uneven bodies (each with its own
        # matrix) under 16 waves, and its all-pairs part alone in 3D
        dict(name="op32_1000", do="op32", geo="lattice", T=1000, kappa=40.0, nrhs=8),
        dict(name="op32_700_sizes", do="op32", geo="sizes", T=700, kappa=20.0, nrhs=16),
        dict(name="g32_100_ellipsoids", do="g32", geo="ellipsoids", T=100, kappa=8.0, nrhs=4),
        # the operator of an FP64 solve, on a ragged size
        dict(name="op64_237", do="op64", geo="lattice", T=237, kappa=40.0, nrhs=5),
        # the scattered field at 4096 targets between the bodies, as the end of the 1000-body workload
        dict(name="field_1000", do="field", geo="lattice", T=1000, kappa=40.0, nrhs=8, M=4096),
        # the field in 3D anywhere outside the MFS surfaces, some targets inside proxies
        dict(name="near_40_ellipsoids", do="near", geo="ellipsoids", T=40, kappa=8.0, nrhs=4, M=3001),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    do = rng.choice(["whole", "solve", "build", "rhs", "op32", "op32", "g32", "op64", "op64", "field", "near"])
    if do == "whole":
        return dict(do=do, geo="star", T=rng.randint(3, 10), kappa=10.0, nrhs=rng.randint(1, 4), M=rng.randint(33, 600), tol=1e-11)
    if do == "solve":
        return dict(do=do, geo="lattice", T=_log(rng, 20, 160), kappa=round(rng.uniform(34, 46), 2), nrhs=rng.randint(1, 8), tol=1e-11)
    if do == "build":
        geo = rng.choice(["lattice", "sizes", "coarse3d"])
        T = {"lattice": _log(rng, 20, 1000), "sizes": _log(rng, 20, 300), "coarse3d": rng.randint(2, 6)}[geo]
        return dict(do=do, geo=geo, T=T, kappa={"lattice": round(rng.uniform(34, 46), 2), "sizes": 20.0, "coarse3d": 3.0}[geo])
    geo = "lattice" if do == "rhs" else rng.choice(["lattice", "lattice", "sizes", "ellipsoids"])
    top = {"lattice": {"op64": 237, "op32": 800, "g32": 800}.get(do, 1000), "sizes": {"op64": 150}.get(do, 500), "ellipsoids": 60 if do.endswith("32") else 25}[geo]
    case = dict(do=do, geo=geo, T=_log(rng, 10, top), nrhs=rng.randint(1, 5) if do == "op64" else rng.randint(1, 8) if not do.endswith("32") else rng.choice([1, 2, 3, 4, 5, 8, 11, 16]),
                kappa={"lattice": round(rng.uniform(34, 46), 2), "sizes": 20.0, "ellipsoids": round(rng.uniform(6, 10), 2)}[geo])
    if do in ("field", "near"):
        case["M"] = _log(rng, 100, 3000)
    return case


# ---------------------------------------------------------------- inputs and calls
def _workload(case, seed):
    T, kappa, nrhs = case["T"], case["kappa"], case.get("nrhs", 1)
    if case["geo"] == "star":
        wl = mi.config0().subset(range(T))
    elif case["geo"] == "lattice":
        wl = mi.config1(seed=seed, T=T, kappa=kappa, nrhs=nrhs)
    elif case["geo"] == "sizes":
        # the sizes are those of T, in an order of the seed's own
        wl = mi.config2(seed=seed, T=T, kappa=kappa, nrhs=nrhs)
        wl.shapes = mi.config2(seed=0, T=T, kappa=kappa, nrhs=nrhs).shapes
        wl.shapes = [wl.shapes[i] for i in np.random.default_rng(seed + 3).permutation(T)]
    elif case["geo"] == "ellipsoids":
        wl = mi.config3(seed=seed, T=T, kappa=kappa)
    else:
        wl = mi.tiny_3d(seed=seed, T=T, kappa=kappa)
    rng = np.random.default_rng(seed + 1)
    if wl.dim == 2:  # plane waves from directions of the seed's own
        a = rng.uniform(0, 2 * math.pi) + 2 * math.pi * np.arange(nrhs) / nrhs
        wl.directions = np.stack([np.cos(a), np.sin(a), 0 * a], axis=1)
    return wl


def _n_sources(wl):
    """Rows of q: every family fixes its shapes' skeleton counts."""
    return sum(wl.shapes[s].k for s in wl.body_shape)


def _cplx(rows, nrhs, seed):
    """Random complex vectors, (rows, nrhs) column-major."""
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return torch.view_as_complex(torch.randn(nrhs, rows, 2, dtype=torch.float64, device=DEV, generator=g)).T


def _targets(case, wl, seed):
    if case["do"] == "field":
        return mi.far_targets(wl, case["M"], seed=seed, mode="gaps")
    # anywhere outside the bodies: two thirds between the proxies, a third between a body and its proxy surface
    M = case["M"]
    far = mi.far_targets(wl, M - M // 3, seed=seed, mode="gaps")
    rng = np.random.default_rng(seed + 2)
    tau = rng.integers(wl.T, size=M // 3)
    rho = np.array([rng.uniform(wl.shapes[s].bound_radius + 0.02, wl.shapes[s].proxy_radius - 0.02) for s in wl.body_shape[tau]])
    e = rng.normal(size=(len(tau), wl.dim))
    near = wl.centres[tau, :wl.dim] + rho[:, None] * e / np.linalg.norm(e, axis=1, keepdims=True)
    return np.concatenate([far, near])


def _device(a):
    return torch.from_numpy(np.ascontiguousarray(a.T)).to(DEV).T


def prepare(case, seed):
    wl, do = _workload(case, seed), case["do"]
    # the option sets of the README and the benchmark; FP64 is the library's default
    opt = dict(precision=mbs.PREC_MIXED, tol=case["tol"], inner_tol=1e-4, restart=200) if do == "solve" else \
        dict(precision=mbs.PREC_MIXED) if do.endswith("32") else dict(tol=case.get("tol", 1e-11))
    state = {"case": case, "wl": wl, "ctx": mbs.Context(wl.dim, wl.kappa, **opt)}
    if do == "build":
        return state
    ctx = state["ctx"].build_scattering_matrices(wl)
    if do in ("whole", "solve", "rhs"):
        state["v"] = _device(wl.boundary_data())
    else:
        state["q"] = _cplx(ctx.N, case["nrhs"], seed)
    if do in ("whole", "field", "near"):
        state["pts"] = _device(_targets(case, wl, seed))
    if do == "near":
        state["qm"] = _cplx(ctx.Nm, case["nrhs"], seed + 7)
    return state


def run(state):
    do, ctx = state["case"]["do"], state["ctx"]
    if do == "build":
        # new geometry: the scattering matrices, and the skeleton that the vectors live on
        ctx.build_scattering_matrices(state["wl"])
        shapes = [ctx.get_shape(s) for s in sorted(set(state["wl"].body_shape.tolist()))]
        return {"S": np.concatenate([s["S"].ravel() for s in shapes]), "skel": np.concatenate([s["skel"] for s in shapes]), "xhat": ctx.get_layout()[2]}
    if do == "rhs":
        return ctx.rhs(state["v"])
    if do == "op32":
        # the single-precision operator: its values carry FP32 accuracy, and a Krylov solver keeps them as complex64
        return ctx.apply_operator(state["q"]).to(torch.complex64)
    if do == "g32":
        return ctx.apply_G(state["q"], mbs.PREC_FP32).to(torch.complex64)
    if do == "op64":
        return ctx.apply_operator(state["q"])
    if do == "field":
        return ctx.evaluate_field(state["pts"], state["q"])
    if do == "near":
        return ctx.evaluate_field_near(state["pts"], state["q"], state["qm"])
    q, _ = ctx.solve(ctx.rhs(state["v"]))
    if do == "solve":
        return q
    # the MFS strengths are an ill-conditioned intermediate; the field that they give is the result
    return {"q": q, "u": ctx.evaluate_field_near(state["pts"], q, ctx.reconstruct(state["v"], q))}


# ---------------------------------------------------------------- floors
def _build_flops(sh):
    m, n, p, k = sh.m, sh.n, sh.p, sh.k
    return 8.0 * (p * (m + n) * min(m, p) + m * n * n + k * m * n + k * k * n)  # the two pivoted factorisations and the products


def work(case):
    wl = _workload(case, 0)
    do, d, r, N, T = case["do"], wl.dim, case.get("nrhs", 1), _n_sources(wl), wl.T
    sh = [wl.shapes[s] for s in wl.body_shape]
    used = [wl.shapes[s] for s in sorted(set(wl.body_shape.tolist()))]
    phi = 35 if d == 2 else 15
    sq = sum(16.0 * s.k ** 2 for s in used)  # the scattering matrices
    pairs = float(N) * N - sum(float(s.k) ** 2 for s in sh)
    M, m, n = case.get("M", 0), sum(s.m for s in sh), sum(s.n for s in sh)
    if do == "build":
        return {"bytes": sum(8.0 * d * (s.m + s.n + s.p) for s in used) + sq + 8.0 * d * N, "flops": sum(map(_build_flops, used))}
    apply_A = sum(8.0 * (s.m * s.n * 2 + s.m * s.k) for s in sh) * r
    one = pairs * (phi + 8.0 * r) + sum(8.0 * s.k ** 2 for s in sh) * r
    vec = 16.0 * N * r
    if do == "rhs":
        return {"bytes": 16.0 * (m * r + sum(2 * s.m * s.n + s.m * s.k for s in used)) + vec, "flops": apply_A}
    if do == "g32":
        return {"bytes": vec + 4.0 * d * N, "flops": pairs * (phi + 8.0 * r)}
    if do in ("op32", "op64"):
        return {"bytes": (2 * vec + sq) / (2 if do == "op32" else 1) + 8.0 * d * N, "flops": one}
    far = float(N) * M * (phi + 8.0 * r)
    if do in ("field", "near"):
        return {"bytes": vec + 16.0 * M * r + 8.0 * d * (N + M) + (16.0 * n * r if do == "near" else 0), "flops": far}
    steps = 20.0 * math.sqrt(T)  # operator applications that such a solve takes, about
    if do == "solve":
        return {"bytes": 16.0 * m * r + vec, "flops": apply_A + steps * one}
    return {"bytes": 16.0 * m * r + vec + 16.0 * M * r, "flops": 2 * apply_A + (steps + 1) * one + far}


# ---------------------------------------------------------------- the same in plain 64-bit torch
def _halves(a):
    t = a * 134217729.0
    hi = t - (t - a)
    return hi, a - hi


def _two_prod(a, b):
    """a * b exactly, as a sum of two (Dekker 1971)."""
    (ah, al), (bh, bl), p = _halves(a), _halves(b), a * b
    return p, ((ah * bh - p) + (ah * bl + al * bh)) + al * bl


def _distance(P, Q):
    """|P_i - Q_j| as r + e, e what rounding left off r."""
    s = e = 0.0
    for c in range(P.shape[1]):
        a, b = P[:, None, c], -Q[None, :, c]
        d = a + b
        t = d - a
        lost = (a - (d - t)) + (b - t)
        p, pe = _two_prod(d, d)
        z = s + p
        t = z - s
        e = e + (s - (z - t)) + (p - t) + pe + 2 * d * lost
        s = z
    r = torch.sqrt(s)
    p, pe = _two_prod(r, r)
    return r, torch.where(r > 0, (((s - p) - pe) + e) / (2 * r), 0 * r)


def _phi(dim, kappa, P, Q):
    """The fundamental solution between all points of P and Q."""
    r, e = _distance(P, Q)
    x, lost = _two_prod(r, kappa)
    turn = torch.polar(torch.ones_like(x), lost + kappa * e)
    if dim == 3:
        return torch.polar(1.0 / (4 * math.pi * r), x) * turn
    near = x < 25
    y = torch.where(near, torch.full_like(x, 25.0), x)
    P0, Q0, a, w = torch.ones_like(y), torch.zeros_like(y), 1.0, 1 / y
    t = torch.ones_like(y)
    for j in range(1, 21):  # Hankel's expansion: sum of i^j a_j / x^j
        a *= -((2 * j - 1) ** 2) / (8.0 * j)
        t = t * w
        if j % 2 == 0:
            P0 = P0 + (1 if j % 4 == 0 else -1) * a * t
        else:
            Q0 = Q0 + (1 if j % 4 == 1 else -1) * a * t
    H = torch.complex(P0, Q0) * torch.polar(torch.sqrt(2 / (math.pi * y)), y) * complex(math.sqrt(0.5), -math.sqrt(0.5))
    if bool(near.any()):
        # Hankel's integral (2 / sqrt(pi)) int_0^inf e^{-s^2} (1 + i s^2 / 2x)^{-1/2} ds by the trapezoidal rule
        z, h = x[near], 0.125
        total = torch.full_like(z, 0.5) + 0j
        for j in range(1, 51):
            total = total + math.exp(-((j * h) ** 2)) / torch.sqrt(torch.complex(torch.ones_like(z), (j * h) ** 2 / (2 * z)))
        H[near] = total * (2 * h / math.sqrt(math.pi)) * torch.polar(torch.sqrt(2 / (math.pi * z)), z) * complex(math.sqrt(0.5), -math.sqrt(0.5))
    return 0.25j * H * turn


def _t(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device=DEV)


def _skeletons(wl, used):
    """Column-pivoted QR of every used shape's B: the first k pivots, ties to the lowest column."""
    P, Mx = max(wl.shapes[s].p for s in used), max(wl.shapes[s].m for s in used)
    B = torch.zeros(len(used), P, Mx, dtype=torch.complex128, device=DEV)
    for i, s in enumerate(used):
        sh = wl.shapes[s]
        B[i, :sh.p, :sh.m] = _phi(wl.dim, wl.kappa, _t(sh.z), _t(sh.x))
    first = torch.arange(Mx, device=DEV)
    at, piv, done = torch.arange(len(used), device=DEV), [], torch.zeros(len(used), Mx, dtype=torch.bool, device=DEV)
    for _ in range(max(wl.shapes[s].k for s in used)):
        n2 = torch.view_as_real(B).square().sum((1, 3)).masked_fill(done, -1.0)
        top = n2.amax(1, keepdim=True)
        # a shape with all columns taken (the others of the batch go on) keeps to a column that is there, and to zeros
        j = torch.where(n2 >= (1 - 1e-10) ** 2 * top, first, Mx).amin(1).clamp_max(Mx - 1)
        v = B[at, :, j] * torch.where(top > 0, top.clamp_min(1e-300).rsqrt(), 0.0)
        B -= v[:, :, None] * torch.einsum("sp,spm->sm", v.conj(), B)[:, None, :]
        done[at, j] = True
        piv.append(j)
    piv = torch.stack(piv, 1).cpu().numpy()
    return {s: piv[i, :wl.shapes[s].k] for i, s in enumerate(used)}


class _Exact:
    def __init__(self, case, seed):
        self.wl = wl = _workload(case, seed)
        used = sorted(set(wl.body_shape.tolist()))
        self.skel = _skeletons(wl, used)
        # world coordinates summed as c + R x, one product at a time
        pts = []
        for t, s in enumerate(wl.body_shape):
            x, R = wl.shapes[s].x[self.skel[s]], wl.rots[t]
            pts.append(np.stack([wl.centres[t, a] + sum(R[a, b] * x[:, b] for b in range(wl.dim)) for a in range(wl.dim)], axis=1))
        self.xhat = _t(np.concatenate(pts))
        self.body = torch.as_tensor(np.repeat(np.arange(wl.T), [len(p) for p in pts]), device=DEV)
        self.off = np.concatenate([[0], np.cumsum([len(p) for p in pts])])
        self.parts = {}

    def rows(self, pts, skip):
        """Blocks of rows of phi(t_i - x_j), zero at the sources of the body skip[i]."""
        step = max(1, 20_000_000 // len(self.xhat))
        for i in range(0, len(pts), step):
            K = _phi(self.wl.dim, self.wl.kappa, pts[i:i + step], self.xhat)
            yield K.masked_fill_(skip[i:i + step, None] == self.body[None, :], 0)

    def sums(self, pts, q, skip):
        return torch.cat([K @ q for K in self.rows(pts, skip)])

    def factors(self, s):
        """Z*, C and the truncated SVD of A of one shape (2D, well-conditioned families)."""
        if s not in self.parts:
            sh, wl = self.wl.shapes[s], self.wl
            x, y, z = _t(sh.x), _t(sh.y), _t(sh.z)
            B, D, A = (_phi(wl.dim, wl.kappa, *p).cpu().numpy() for p in ((z, x), (z, y), (x, y)))
            Q, R = np.linalg.qr(B[:, self.skel[s]])
            Zs = np.linalg.solve(R, Q.conj().T @ B)
            (U, g, V), (u, h, w) = (np.linalg.svd(M, full_matrices=False) for M in (A, B))
            r, n = int(np.sum(g > 1e-14 * g[0])), int(np.sum(h > 1e-14 * h[0]))
            U, g, V = U[:, :r], g[:r], V[:r]
            C = w[:n].conj().T @ ((u[:, :n].conj().T @ D) / h[:n, None])
            S = ((Zs @ C) @ V.conj().T / g) @ (U.conj().T @ Zs.T)
            self.parts[s] = [torch.as_tensor(a, device=DEV) for a in (Zs, C, U, g, V.conj().T.copy(), S)]
        return self.parts[s]

    def each(self, f):
        return torch.cat([f(t, int(s)) for t, s in enumerate(self.wl.body_shape)])

    def pinv(self, s, t):
        _, _, U, g, V, _ = self.factors(s)
        return V @ ((U.conj().T @ t) / g[:, None])

    def v_of(self, v, t):
        o = np.concatenate([[0], np.cumsum(self.wl.m_of_body())])
        return v[o[t]:o[t + 1]]

    def rhs(self, v):
        return self.each(lambda t, s: self.factors(s)[0] @ (self.factors(s)[1] @ self.pinv(s, self.v_of(v, t))))

    def S_times(self, y):
        return self.each(lambda t, s: self.factors(s)[5] @ y[self.off[t]:self.off[t + 1]])

    def solve(self, b):
        A = self.S_times(torch.cat(list(self.rows(self.xhat, self.body))))
        A.diagonal().add_(1.0)
        return torch.linalg.solve(A, b)

    def mfs(self, pts, tau, qm):
        """The fields of the bodies tau at their own targets (tau < 0: none) from their MFS sources."""
        wl = self.wl
        u = torch.zeros(len(pts), qm.shape[1], dtype=torch.complex128, device=DEV)
        o = np.concatenate([[0], np.cumsum([wl.shapes[s].n for s in wl.body_shape])])
        for t in sorted(set(tau.tolist()) - {-1}):
            at = torch.as_tensor(np.nonzero(tau == t)[0], device=DEV)
            u[at] = _phi(wl.dim, wl.kappa, pts[at], _t(wl.body_points(t, "y"))) @ qm[o[t]:o[t + 1]]
        return u


def exact(case, seed):
    do = case["do"]
    if do == "build" or (do in ("op32", "op64") and case["geo"] != "lattice"):
        return None  # scattering matrices of these bodies are defined only to the conditioning of the MFS, far above rounding
    E = _Exact(case, seed)
    wl = E.wl
    if do in ("whole", "solve", "rhs"):
        v = torch.as_tensor(wl.boundary_data(), device=DEV)
        b = E.rhs(v)
        if do == "rhs":
            return b
        q = E.solve(b)
        if do == "solve":
            return q
    else:
        q = _cplx(_n_sources(wl), case["nrhs"], seed).contiguous()
    if do in ("op32", "op64", "g32"):
        y = E.sums(E.xhat, q, E.body)
        return y if do == "g32" else q + E.S_times(y)
    P = _targets(case, wl, seed)
    pts = _t(P)
    if do == "field":
        return E.sums(pts, q, torch.full((len(P),), -1, device=DEV))
    d2 = ((P[:, None, :] - wl.centres[None, :, :wl.dim]) ** 2).sum(2)
    inside = d2 < wl.proxy_radius_of_body()[None, :] ** 2
    tau = np.where(inside.any(1), inside.argmax(1), -1)
    if do == "whole":
        w = E.sums(E.xhat, q, E.body)
        qm = E.each(lambda t, s: E.pinv(s, E.v_of(v, t) - E.factors(s)[0].T @ w[E.off[t]:E.off[t + 1]]))
    else:
        qm = _cplx(sum(wl.shapes[s].n for s in wl.body_shape), case["nrhs"], seed + 7).contiguous()
    u = E.sums(pts, q, torch.as_tensor(tau, device=DEV)) + E.mfs(pts, tau, qm)
    return {"q": q, "u": u} if do == "whole" else u
