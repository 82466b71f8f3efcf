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
