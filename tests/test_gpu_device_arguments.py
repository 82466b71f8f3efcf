"""CUDA tensors that torch is still computing when they are passed: every call
takes their finished values, whatever stream they are made on and whatever
stream the context runs on."""
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


@pytest.mark.parametrize("maker", ["default", "side"])
@pytest.mark.parametrize("runner", ["own", "given"])
def test_arguments_in_the_making(pkg, maker, runner):
    """Row-major tensors (the binding copies them on torch's stream) filled behind
    50 ms of queued work give the results of host arrays, to the bit."""
    import torch
    wl = mi.tiny_2d(seed=1, T=9, kappa=6.0, nrhs=3)
    given = torch.cuda.Stream()
    kw = {"stream": given.cuda_stream} if runner == "given" else {}
    with pkg.Context(2, wl.kappa, **kw) as ctx:
        ctx.build_scattering_matrices(wl)
        rng = np.random.default_rng(0)
        far = mi.far_targets(wl, 300, seed=5, mode="gaps")
        near = far.copy()
        near[::3] = wl.centres[2, :2]
        near[::3, 0] += 0.9 * wl.proxy_radius_of_body()[2]
        q, qm, v = (rng.normal(size=(n, 3)) + 1j * rng.normal(size=(n, 3)) for n in (ctx.N, ctx.Nm, ctx.Mtot))
        calls = [
            (ctx.evaluate_field, (far, q)), (ctx.evaluate_field_near, (near, q, qm)), (ctx.rhs, (v,)),
            (ctx.apply_operator, (q,)), (ctx.apply_G, (q,)), (ctx.reconstruct, (v, q)),
            (lambda b: ctx.solve(b)[0], (q,)),
        ]
        stream = torch.cuda.default_stream() if maker == "default" else torch.cuda.Stream()
        for f, args in calls:
            want = f(*args)
            ready = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in args]
            late = [torch.zeros_like(a) for a in ready]
            torch.cuda.synchronize()
            with torch.cuda.stream(stream):
                torch.cuda._sleep(100_000_000)
                for a, b in zip(late, ready):
                    a.copy_(b)
                got = f(*late)
            torch.cuda.synchronize()
            assert np.array_equal(got.cpu().numpy(), want)


def test_beside_a_context_that_captures_on_a_blocking_stream(pkg):
    """One thread solves on a stream of the kind that the default stream waits for,
    its steps captured as graphs; another passes device arguments all the while."""
    import ctypes
    import threading
    import torch
    wl = mi.tiny_2d(seed=1, T=9, kappa=6.0, nrhs=3)
    rt = ctypes.CDLL("libcudart.so.13")
    st = ctypes.c_void_p()
    assert rt.cudaStreamCreate(ctypes.byref(st)) == 0
    failed, done = [], threading.Event()
    with pkg.Context(2, wl.kappa, stream=st.value, restart=30, tol=1e-10) as a, pkg.Context(2, wl.kappa) as b:
        a.build_scattering_matrices(wl)
        b.build_scattering_matrices(wl)
        rhs = a.rhs(wl.boundary_data())
        q = torch.from_numpy(np.ascontiguousarray(rhs.T)).cuda().T
        want = b.apply_G(rhs)

        def solve():
            try:
                for _ in range(20):
                    a.set_options(tol=1e-10)  # drops the captured steps
                    a.solve(rhs, raise_on_noconv=False)
            except Exception as e:
                failed.append(e)
            done.set()

        t = threading.Thread(target=solve)
        t.start()
        got = []
        while not done.is_set():  # no torch work in between: its default stream minds captures too
            got.append(b.apply_G(q))
        t.join()
        assert not failed and len(got) > 20
        assert all(np.array_equal(y.cpu().numpy(), want) for y in got)
    assert rt.cudaStreamDestroy(st) == 0
