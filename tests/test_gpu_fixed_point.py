"""GPU kernels beside the general ones: the fixed-point sums (gfixed.cu), the
S build shared out over clusters, the blocked right-hand side, the sorting of
targets to proxies and the Gram-Schmidt updates on clusters, at the sizes where
each can go wrong."""
import numpy as np
import pytest

import mbs_inputs as mi
import oracle as orc

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_2603_19113_gb300 as p
    return p


def _rand(shape, seed):
    rng = np.random.default_rng(seed)
    return rng.normal(size=shape) + 1j * rng.normal(size=shape)


def _rel(a, b):
    return float(np.max(np.abs(a - b)) / np.max(np.abs(b)))


def _ctx(pkg, wl, **kw):
    ctx = pkg.Context(wl.dim, wl.kappa, **kw)
    ctx.build_scattering_matrices(wl)
    N, off, x = ctx.get_layout()
    body = np.repeat(np.arange(wl.T), np.diff(off))
    return ctx, x, body, off


# 9 bodies: 4 groups of threads a target; 90: one; kappa = 0.9: pairs below
# kappa r = 4; 3D bodies of 70 points: three rounds of 32 sources, the last ragged
_WL = {
    "2d": lambda: mi.tiny_2d(seed=1, T=9, kappa=6.0, ks=(24, 37, 50)),
    "2d_90": lambda: mi.tiny_2d(seed=3, T=90, kappa=9.0, ks=(24, 33, 65)),
    "2d_low": lambda: mi.tiny_2d(seed=2, T=9, kappa=0.9, ks=(30, 41)),
    "2d_high": lambda: mi.tiny_2d(seed=4, T=9, kappa=30.0, ks=(24, 37, 50)),
    "3d": lambda: mi.tiny_3d(seed=0, T=5, kappa=3.0, nth=10, nph=14, p=141, k=70),
}


@pytest.mark.parametrize("case,nrhs", [(c, n) for c in _WL for n in (1, 6)] + [("2d", n) for n in (2, 3, 4, 5, 7, 8, 9, 17)]
                         + [("3d", n) for n in (3, 8)])
def test_fixed_point_sums(pkg, case, nrhs):
    """Ghat q and the field at targets against the oracle and the FP64-pipe kernel
    (bound of the FP64 kernels: rounding of sums of N terms accurate to ~1e-15)."""
    wl = _WL[case]()
    ctx, x, body, _ = _ctx(pkg, wl)
    q = _rand((ctx.N, nrhs), nrhs)
    ref = orc.G_dense(wl.dim, wl.kappa, x, body) @ q
    y = ctx.apply_G(q)
    assert _rel(y, ref) < 1e-12
    t = mi.far_targets(wl, 131, seed=3, mode="gaps")
    u = ctx.evaluate_field(t, q)
    assert _rel(u, orc.field(wl.dim, wl.kappa, t, x, q)) < 1e-12
    ctx.set_options(fp64_kernel=0)
    assert _rel(y, ctx.apply_G(q)) < 1e-12
    assert _rel(u, ctx.evaluate_field(t, q)) < 1e-12


def test_fixed_point_scales_and_non_finite_entries(pkg):
    """Bodies of very different magnitude keep their own scale; entries beyond
    it, infinities and NaN take the FP64 sums: they reach every other body and
    leave their own alone."""
    wl = _WL["2d"]()
    ctx, x, body, off = _ctx(pkg, wl)
    G = orc.G_dense(2, wl.kappa, x, body)
    q = _rand((ctx.N, 2), 5)
    q[body == 1] *= 1e-200
    q[body == 2] = 0.0
    q[body == 3] *= 1e150
    for only in range(wl.T):
        qq = np.where((body == only)[:, None], q, 0)
        ref = G @ qq
        y = ctx.apply_G(qq)
        if only == 2:
            assert not y.any()
        else:
            assert _rel(y, ref) < 1e-12
    for value in (1e-300, 1e290, np.nan, np.inf):
        qq = _rand((ctx.N, 2), 6)
        qq[off[4] + 3, 1] = value
        y = ctx.apply_G(qq)
        if np.isfinite(value):
            ctx.set_options(fp64_kernel=0)
            ref = ctx.apply_G(qq)
            assert all(_rel(y[:, r], ref[:, r]) < 1e-12 for r in (0, 1))
            ctx.set_options(fp64_kernel=2)
        else:
            assert np.isfinite(y[:, 0]).all()
            assert np.array_equal(np.isfinite(y[:, 1]), body == 4)


def test_fixed_point_gives_way_when_memory_runs_out(pkg):
    """The smallest budget at which the FP64-pipe kernel's operator runs is
    enough for the default one too: it then runs without its own workspace."""
    wl = _WL["2d_90"]()

    def run(budget, kernel):
        try:
            with pkg.Context(2, wl.kappa, hbm_budget=budget, fp64_kernel=kernel) as ctx:
                ctx.build_scattering_matrices(wl)
                return ctx.apply_G(_rand((ctx.N, 17), 1))
        except pkg.MbsError as e:
            assert e.status == 3  # out of memory
            return None

    lo, hi = 1, 1 << 28
    while hi - lo > 4096:
        mid = (lo + hi) // 2
        lo, hi = (mid, hi) if run(mid, 0) is None else (lo, mid)
    y = run(hi, 2)
    assert y is not None
    assert _rel(y, run(hi, 0)) < 1e-12
    assert _rel(run(1 << 28, 2), y) < 1e-12


@pytest.mark.parametrize("make", [lambda k: mi.shape_2d("star3n", 2 * k, k, 2 * k + 1, 1.3, k=k),
                                  lambda k: mi.shape_ellipsoid(0.9, 0.7, 0.8, nth=8, nph=2 * -(-k // 4), p=141, k=k)])
def test_S_does_not_depend_on_the_team(pkg, make):
    """One shape on a cluster of 8 CTAs, among 30 on clusters of 4, and among 160
    on one CTA each: the same matrix to the bit (odd and even sizes, B of full
    and of lower rank)."""
    shapes = [make(k) for k in (24, 37, 50)]
    dim, kappa = shapes[0].dim, 6.0

    def S_of(copies):
        T = copies * len(shapes)
        side = int(np.ceil(T ** (1 / dim)))
        grid = np.stack(np.meshgrid(*[np.arange(side)] * dim, indexing="ij"), -1).reshape(-1, dim)[:T]
        centres = np.zeros((T, 3))
        centres[:, :dim] = 4.0 * grid
        wl = mi.Workload("team", dim, kappa, shapes * copies, np.arange(T, dtype=np.int32), centres,
                         np.repeat(np.eye(3)[None], T, axis=0), np.array([[1.0, 0, 0]]))
        with pkg.Context(dim, kappa) as ctx:
            ctx.build_scattering_matrices(wl)
            return [ctx.get_shape(s) for s in range(T)]

    one = S_of(1)
    for copies in (10, 54):
        for s, got in enumerate(S_of(copies)):
            assert np.array_equal(got["skel"], one[s % 3]["skel"])
            assert np.array_equal(got["S"], one[s % 3]["S"]), (copies, s)


@pytest.mark.parametrize("ks,m_per_k", [((24, 37, 64), 2), ((24, 37, 65), 2), ((24, 37, 51), 5), ((24, 37, 52), 5)])
@pytest.mark.parametrize("nrhs", [1, 8, 11])
def test_rhs_blocks(pkg, ks, m_per_k, nrhs):
    """b from blocks of 8 right-hand sides (128, 130, 255 points in the largest
    body) and beyond them (260): the columns one by one to the bit, and the
    oracle's within 1e-9 (3e-11 is what an oracle whose points carry one rounding
    differs from the oracle by, at most)."""
    kappa = 15.0
    wl = mi.tiny_2d(seed=5, T=4, kappa=kappa, nrhs=nrhs, ks=ks, m_per_k=m_per_k)
    with pkg.Context(2, kappa) as ctx:
        ctx.build_scattering_matrices(wl)
        v = wl.boundary_data()
        b = ctx.rhs(v)
        for r in range(nrhs):
            assert np.array_equal(ctx.rhs(v[:, r]), b[:, r])
        xhat = ctx.get_layout()[2]
    t = mi.far_targets(wl, 64, mode="ring")
    sdata = orc.build_all(wl)
    lay = orc.layout(wl, sdata)
    # compared through the field they radiate: b itself is defined to the noise of the ID
    got = orc.field(2, kappa, t, xhat, b)
    ref = orc.field(2, kappa, t, lay["xhat"], orc.rhs(wl, sdata, lay, v))
    assert _rel(got, ref) < 1e-9


@pytest.mark.parametrize("dim", [2, 3])
@pytest.mark.parametrize("M", [1, 127, 300])
def test_targets_are_sorted_to_proxies(pkg, dim, M):
    """The first target inside a proxy is reported, targets on its outside pass,
    non-finite ones are refused before anything else; host and device targets."""
    import torch
    wl = mi.tiny_2d(seed=1, T=9, kappa=6.0) if dim == 2 else mi.tiny_3d(seed=0, T=5, kappa=3.0, nth=10, nph=14, p=141, k=70)
    ctx, x, body, _ = _ctx(pkg, wl)
    q = _rand((ctx.N, 1), 1)
    t = mi.far_targets(wl, M, seed=5, mode="gaps")
    pr = wl.proxy_radius_of_body()
    e = np.zeros(dim)
    e[0] = 1.0
    t[-1] = wl.centres[2, :dim] + pr[2] * (1 + 1e-9) * e
    u = ctx.evaluate_field(t, q)
    dev = torch.from_numpy(np.ascontiguousarray(t.T)).cuda().T
    ud = ctx.evaluate_field(dev, torch.from_numpy(np.ascontiguousarray(q.T)).cuda().T)
    assert np.array_equal(ud.cpu().numpy(), u)
    bad = t.copy()
    i = M // 2
    bad[i] = wl.centres[2, :dim] + pr[2] * (1 - 1e-9) * e
    bad[-1] = wl.centres[1, :dim]
    with pytest.raises(pkg.MbsError) as err:
        ctx.evaluate_field(bad, q)
    assert err.value.status == 7 and f"target {min(i, M - 1)} lies inside the proxy surface of body {2 if i < M - 1 else 1}" in str(err.value)
    bad[0] = np.nan
    with pytest.raises(pkg.MbsError) as err:
        ctx.evaluate_field(bad, q)
    assert err.value.status == 1
    # the field inside a proxy leaves out that body's skeleton: its MFS sources alone carry it
    qm = _rand((ctx.Nm, 1), 2)
    near = t.copy()
    near[i] = wl.centres[2, :dim] + 0.9 * pr[2] * e
    un = ctx.evaluate_field_near(near, q, qm)
    K = orc.kernel_matrix(dim, wl.kappa, near[i:i + 1], x)
    K[:, body == 2] = 0
    n_of = [wl.shapes[s].n for s in wl.body_shape]
    o = int(np.sum(n_of[:2]))
    ref = K @ q + orc.kernel_matrix(dim, wl.kappa, near[i:i + 1], wl.body_points(2, "y")) @ qm[o:o + n_of[2]]
    assert _rel(un[i:i + 1], ref) < 1e-12


@pytest.mark.parametrize("T,ks", [(30, (24, 36, 50)), (300, (50,)), (460, (64,))])
def test_basis_update_teams(pkg, T, ks):
    """Mixed solves whose Gram-Schmidt updates run on clusters of 4, 2 and 1 CTAs
    per row tile (16 rows ragged, and bases from one column block up): the residual
    the solver reports is the one its FP64 operator shows, and refinement contracts
    as an exact Arnoldi relation lets it."""
    wl = mi.tiny_2d(seed=6, T=T, kappa=12.0, nrhs=8, ks=ks)
    with pkg.Context(2, wl.kappa, precision=pkg.PREC_MIXED, tol=1e-11, restart=100) as ctx:
        ctx.build_scattering_matrices(wl)
        b = ctx.rhs(wl.boundary_data())
        q, info = ctx.solve(b)
        assert info["converged"] == 1 and info["fp64_finish"] == 0 and info["sweeps"] <= 4
        ctx.set_options(precision=pkg.PREC_FP64)
        r = b - ctx.apply_operator(q)
        assert np.max(np.linalg.norm(r, axis=0) / np.linalg.norm(b, axis=0)) < 1e-11 * 1.01


@pytest.mark.parametrize("T,kappa,kernel", [(160, 0.25, 1), (160, 40.0, 2), (12, 0.25, 2)])
def test_kernel_of_a_low_frequency_solve(pkg, T, kappa, kernel):
    """Double-float where the tolerance allows it and the formats leave out four in
    five body pairs (160 bodies, kappa = 0.25: 20 ms a launch, fixed point 33)."""
    wl = mi.config1(seed=0, T=T, kappa=kappa, nrhs=8)
    with pkg.Context(2, kappa, precision=pkg.PREC_MIXED, tol=1e-9, restart=200) as ctx:
        ctx.build_scattering_matrices(wl)
        b = ctx.rhs(wl.boundary_data())
        q, info = ctx.solve(b)
        assert info["converged"] == 1 and info["fp64_kernel"] == kernel
        ctx.set_options(precision=pkg.PREC_FP64, fp64_kernel=0)
        r = b - ctx.apply_operator(q)
        assert np.max(np.linalg.norm(r, axis=0) / np.linalg.norm(b, axis=0)) < 1e-9 * 1.01
        if kernel == 1:  # a tolerance that double-float does not reach
            ctx.set_options(precision=pkg.PREC_MIXED, fp64_kernel=2, tol=1e-13, max_iter=3)
            assert ctx.solve(b, raise_on_noconv=False)[1]["fp64_kernel"] == 2


@pytest.mark.parametrize("case", ["2d", "2d_high", "2d_low", "3d", "3d_low"])
@pytest.mark.parametrize("nrhs", [1, 8])
def test_fixed_point_accuracy(pkg, case, nrhs):
    """Sampled rows against 30-digit sums over the same coordinates.  A pair is off
    by 1e-15 in phi and its product, by kappa 2^-53 through the rounding of a source's
    offset (radius 1) and by kappa 2^e 2^-58 <= kappa 2^-54 in the phase, pairs of
    different sources independently: five times the root of the sum of their squares."""
    mp = pytest.importorskip("mpmath")
    mp.mp.dps = 30
    wl = mi.tiny_3d(seed=0, T=5, kappa=0.5, nth=10, nph=14, p=141, k=70) if case == "3d_low" else _WL[case]()
    ctx, x, body, off = _ctx(pkg, wl)
    q = _rand((ctx.N, nrhs), 4)
    y = ctx.apply_G(q)
    for i in np.linspace(0, ctx.N - 1, 5).astype(int):
        phi = []
        for j in range(ctx.N):
            r = mp.sqrt(sum((mp.mpf(float(a)) - mp.mpf(float(b))) ** 2 for a, b in zip(x[i], x[j])))
            phi.append(mp.mpc(0) if body[i] == body[j] else mp.mpc(0, 0.25) * mp.hankel1(0, wl.kappa * r) if wl.dim == 2 else
                       mp.exp(mp.mpc(0, wl.kappa) * r) / (4 * mp.pi * r))
        for c in range(nrhs):
            ref = mp.fsum(p * mp.mpc(complex(v)) for p, v in zip(phi, q[:, c]))
            size = float(mp.sqrt(mp.fsum(abs(p) ** 2 * abs(v) ** 2 for p, v in zip(phi, q[:, c].tolist()))))
            assert abs(mp.mpc(complex(y[i, c])) - ref) < 5 * size * (1e-15 + wl.kappa * (2.0 ** -53 + 2.0 ** -54))


def _scaled(wl, s):
    import dataclasses
    shapes = [dataclasses.replace(h, x=h.x * s, y=h.y * s, z=h.z * s, proxy_radius=h.proxy_radius * s,
                                  bound_radius=h.bound_radius * s) for h in wl.shapes]
    return dataclasses.replace(wl, kappa=wl.kappa / s, shapes=shapes, centres=wl.centres * s)


@pytest.mark.parametrize("e", [-75, -70, -62, 62, 70])
def test_sums_in_any_unit_of_length(pkg, e):
    """2D sums depend on kappa times lengths alone: the FP64-accurate ones of a
    geometry 2^e times as large, where squares leave FP32's range too."""
    wl = _WL["2d"]()
    ctx, x, body, _ = _ctx(pkg, wl)
    big, xb, _, _ = _ctx(pkg, _scaled(wl, 2.0 ** e))
    if not np.array_equal(xb, x * 2.0 ** e):
        pytest.skip("another skeleton")
    q = _rand((ctx.N, 3), 1)
    assert _rel(big.apply_G(q), ctx.apply_G(q)) < 1e-12


@pytest.mark.parametrize("T,nrhs,ks,m_per_k", [
    (160, 3, (24, 37, 64), 2),   # 2 right-hand sides a CTA would take 320 CTAs: 3 a CTA
    (50, 6, (24, 37, 64), 2),    # 2 a CTA
    (40, 7, (24, 37, 64), 2),    # 4 a CTA, the last 3
    (160, 11, (24, 37, 64), 2),  # 8 a CTA, the last 3; one column alone: the general kernel
    (80, 8, (24, 37, 65), 2),    # 130 points: 8 row groups
    (64, 11, (24, 37, 51), 5),   # 255 points
    (64, 11, (24, 48, 64), 4),   # 256 points
])
def test_blocked_rhs_and_reconstruction(pkg, T, nrhs, ks, m_per_k):
    """Several right-hand sides a CTA (152 SMs) give each column what it gets alone,
    where it takes another kernel or another share of a CTA: to the bit."""
    wl = mi.tiny_2d(seed=5, T=T, kappa=15.0, nrhs=nrhs, ks=ks, m_per_k=m_per_k)
    with pkg.Context(2, wl.kappa) as ctx:
        ctx.build_scattering_matrices(wl)
        v, q = wl.boundary_data(), _rand((ctx.N, nrhs), 3)
        b, qm = ctx.rhs(v), ctx.reconstruct(v, q)
        for r in range(nrhs):
            assert np.array_equal(ctx.rhs(v[:, r]), b[:, r])
            assert np.array_equal(ctx.reconstruct(v[:, r], q[:, r]), qm[:, r])


def test_fixed_point_sums_at_full_size(pkg):
    """The bench workload's 256 sampled rows through the default kernel."""
    from test_gpu_parity import test_G_full_size_config1_sampled_rows as full_size
    full_size(pkg, 0, 2)
