"""The launch-shape autotuner of the FP32 G_hat: which kernel it takes, what it
costs, and that its trials cost no other call its memory."""
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


def _rand(shape, seed):
    rng = np.random.default_rng(seed)
    return rng.normal(size=shape) + 1j * rng.normal(size=shape)


def test_kernel_and_cost_of_a_class(pkg):
    """19 bodies of 300 points, 11 right-hand sides: the tensor cores are a tenth
    faster (213 and 238 us) and taken.  Trials: two kernels, each launched once
    untimed, two or three counts a kernel and three more of the one taken, each
    at most three times; a launch is packing or none, one or two passes and the
    reduction: 4 * 2 + 8 * 3 * 4 = 104 kernels at most, and 4 for the call."""
    wl = mi.config3(seed=1, T=19, kappa=8.0)
    with pkg.Context(3, wl.kappa) as ctx:
        ctx.build_scattering_matrices(wl)
        q = _rand((ctx.N, 11), 1)
        n0 = pkg.launch_count()
        ctx.apply_G(q, pkg.PREC_FP32)
        assert pkg.launch_count() - n0 <= 108
        assert ctx.kernel_times()["g32_path"] == 3
        # of launches beyond 0.2 ms each is timed once
        wl = mi.config3(seed=1, T=40, kappa=8.0)
        ctx.build_scattering_matrices(wl)
        q = _rand((ctx.N, 11), 1)
        n0 = pkg.launch_count()
        ctx.apply_G(q, pkg.PREC_FP32)
        assert pkg.launch_count() - n0 <= 2 * 4 + 8 * 4 + 4 + 2


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


def test_trials_leave_the_fixed_point_workspace_alone(pkg):
    """A budget that holds the FP32 operator at its usual shape and the fixed-point
    kernel's workspace holds both after the trials of a class of its own."""
    wl = mi.tiny_2d(seed=3, T=200, kappa=9.0, nrhs=13, ks=(24, 33, 65))

    def kernel(budget, autotune):
        with pkg.Context(2, wl.kappa, hbm_budget=budget, autotune=autotune, restart=1, max_iter=1) as ctx:
            ctx.build_scattering_matrices(wl)
            q = _rand((ctx.N, 13), 1)
            ctx.apply_G(q)
            ctx.apply_G(q, pkg.PREC_FP32)
            k = ctx.solve(q, raise_on_noconv=False)[1]["fp64_kernel"]
            return k == 2

    least = _least(pkg, lambda b: kernel(b, 0))
    assert kernel(least + 8192, 1)


def test_a_class_tuned_with_more_memory(pkg):
    """The counts that a context without a budget chose are no condition for one
    that has memory for the usual ones, whichever call comes first."""
    wl = mi.tiny_2d(seed=3, T=200, kappa=9.0, nrhs=12, ks=(24, 33, 65))

    def run(budget, autotune, fx_first=True):
        with pkg.Context(2, wl.kappa, hbm_budget=budget, autotune=autotune) as ctx:
            ctx.build_scattering_matrices(wl)
            q = _rand((ctx.N, 12), 1)
            return [ctx.apply_G(q, p) for p in ((pkg.PREC_FP32, pkg.PREC_FP64) if not fx_first else (pkg.PREC_FP64, pkg.PREC_FP32))]

    for fx_first in (True, False):
        ref = run(0, 1, fx_first)
        least = _least(pkg, lambda b: bool(run(b, 0, fx_first)))
        got = run(least + 8192, 1, fx_first)
        for a, b in zip(got, ref):
            assert np.abs(a - b).max() < 2e-5 * np.abs(b).max()
