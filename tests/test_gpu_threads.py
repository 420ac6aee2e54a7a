"""A handle and its clones, each on a host thread and a stream of its own, whose first calls
build what they share (tables of the transforms, the preconditioner's) at the same time as the
others allocate their own arrays.  The same kernels as on one thread, hence the same bits.
"""
import threading

import numpy as np
import pytest

from paper_2403_19854_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2403_19854_gb300 import rk  # noqa: E402

DEV = torch.device("cuda:0")


def calls(p):
    r, g = torch.as_tensor(p.r, device=DEV), torch.as_tensor(p.g, device=DEV)
    x = torch.as_tensor(W.random_field(p.nbox, 3), device=DEV)
    torch.cuda.synchronize()
    kw = dict(tol=1e-9, max_iter=200, raise_on_error=False)

    def explicit(H):
        d = r.clone()
        H.transient_explicit(torch.zeros_like(r), g, 1e-6, 2, d)
        return d, H.apply_precond(x)

    return [lambda H: H.solve(r, g, precision="fp64", **kw)[:2],
            lambda H: H.solve(r, g, precision="mixed", precond="spectral", **kw)[:2],
            lambda H: (H.nonlinear_grad_force(x, "cubic", 0.7, [1.0, 0.5, 0.25]),),
            lambda H: H.solve(r, g, precision="fp64", precond="spectral", **kw)[:2],
            explicit,
            lambda H: (H.apply_precond(x.float()), H.apply_K(x))]


def run(fn, H, out, k, barrier):
    try:
        with torch.cuda.stream(torch.cuda.Stream(device=DEV)):
            barrier.wait()
            out[k] = fn(H)
            torch.cuda.current_stream().synchronize()
    except Exception as e:  # reported by the test
        out[k] = e


@pytest.mark.parametrize("a", [2.0, 5.5])
def test_first_use_on_several_threads(a):
    p = W.cube_problem(36, a, 1, "sin")
    p.g = np.where(p.chi_gamma > 0, 0.1, 0.0)
    fns = calls(p)
    ref = []
    for fn in fns:
        H = rk.Handle.from_problem(p, device=DEV)
        ref.append(fn(H))
        torch.cuda.synchronize()
    for _ in range(4):
        H = rk.Handle.from_problem(p, device=DEV)
        hs = [H] + [H.clone() for _ in fns[1:]]
        out, barrier = [None] * len(fns), threading.Barrier(len(fns))
        ts = [threading.Thread(target=run, args=(fn, h, out, k, barrier)) for k, (fn, h) in enumerate(zip(fns, hs))]
        for t in ts:
            t.start()
        for t in ts:
            t.join()
        for k, (got, want) in enumerate(zip(out, ref)):
            assert not isinstance(got, Exception), (k, got)
            for x, y in zip(got, want):
                assert torch.equal(x, y), k
