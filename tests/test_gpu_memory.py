"""The fixed-point kernel's workspace under a device-memory budget: optional
memory, which refuses no call and is taken up again when there is room."""
import functools

import numpy as np
import pytest

import mbs_inputs as mi

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


@functools.lru_cache(None)
def _wl(T, nrhs=5):
    return mi.tiny_2d(seed=3, T=T, kappa=9.0, nrhs=nrhs, ks=(24, 33, 65))


def _rand(shape, seed):
    rng = np.random.default_rng(seed)
    return rng.normal(size=shape) + 1j * rng.normal(size=shape)


def _least(pkg, works, hi=1 << 31):
    """The smallest budget (to 8 KB) for which works(budget) is true."""
    def ok(budget):
        try:
            return works(budget)
        except pkg.MbsError as e:
            assert e.status == 3  # out of memory
            return False
    lo = 1
    assert ok(hi)
    while hi - lo > 8192:
        mid = (lo + hi) // 2
        lo, hi = (lo, mid) if ok(mid) else (mid, hi)
    return hi


def test_what_fits_beside_the_fp64_pipe_fits(pkg):
    """A budget that a sequence of calls just fits on the FP64 pipe holds it with
    the default kernel: its partial sums and packed sources give way."""
    wl = _wl(90)
    t = mi.far_targets(wl, 2000, seed=3, mode="gaps")

    def calls(budget, kernel):
        with pkg.Context(2, wl.kappa, hbm_budget=budget, fp64_kernel=kernel, restart=20, max_iter=40) as ctx:
            ctx.build_scattering_matrices(wl)
            q = _rand((ctx.N, 5), 1)
            out = [ctx.apply_G(q), ctx.evaluate_field(t[:300], q), ctx.evaluate_field(t, q)]
            ctx.solve(q, raise_on_noconv=False)
            return out + [ctx.apply_G(_rand((ctx.N, 17), 2)), ctx.evaluate_field(t, q)]

    least = _least(pkg, lambda b: bool(calls(b, 0)))
    for a, b in zip(calls(least + 8192, 2), calls(least, 0)):
        assert np.abs(a - b).max() < 1e-12 * np.abs(b).max()


def test_the_workspace_comes_back(pkg):
    """After a build that needed its memory, and with a larger budget."""
    wl = _wl(9)

    def solve(ctx):
        return ctx.solve(_rand((ctx.N, 5), 1), raise_on_noconv=False)[1]["fp64_kernel"]

    def solves(budget, builds, restart):
        with pkg.Context(2, wl.kappa, hbm_budget=budget, restart=restart, max_iter=40) as ctx:
            return [solve(ctx.build_scattering_matrices(wl)) for _ in range(builds)]

    least = _least(pkg, lambda b: solves(b, 2, 20)[0] == 2)
    assert solves(least, 2, 20) == [2, 2]
    least = _least(pkg, lambda b: bool(solves(b, 1, 200)))
    with pkg.Context(2, wl.kappa, hbm_budget=least, restart=200, max_iter=40) as ctx:
        ctx.build_scattering_matrices(wl)
        assert solve(ctx) != 2
        ctx.set_options(hbm_budget=0)
        assert solve(ctx) == 2
