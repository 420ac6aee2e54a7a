"""Handles used again: the captured chunk of CG iterations of a batched solve belongs to the
steps it was captured with, and what an earlier call left in the work arrays is not read.  The
same kernels in the same order as on new handles, hence the same bits.
"""
import numpy as np
import pytest

from paper_2403_19854_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2403_19854_gb300 import rk  # noqa: E402

DEV = torch.device("cuda:0")


def batch(p, sources):
    H = rk.Handle.from_problem(p, device=DEV)
    hs = [H] + [H.clone() for _ in sources[1:]]
    new = lambda: torch.empty(p.nbox, dtype=torch.float64, device=DEV)  # noqa: E731
    t = lambda v: torch.as_tensor(v, device=DEV)  # noqa: E731
    return [(h, t(r), t(p.g), new(), new()) for h, r in zip(hs, sources)]


def solve(items, precond):
    infos = rk.solve_batched(items, precision="mixed", tol=1e-10, precond=precond)
    return [(i["status"], i["iterations"], it[3].cpu().numpy(), it[4].cpu().numpy()) for i, it in zip(infos, items)]


@pytest.mark.parametrize("order", [("none", "spectral", "none"), ("spectral", "none", "spectral")], ids="-".join)
def test_batched_again_with_another_preconditioner(order):
    p = W.cube_problem(48, 2.0, 1, "sin")
    p.g = np.where(p.chi_gamma > 0, 0.1, 0.0)
    sources = [p.r, np.where(p.chi > 0, W.random_field(p.nbox, 5), 0.0)]
    fresh = {k: solve(batch(p, sources), k) for k in set(order)}
    items = batch(p, sources)
    for precond in order:
        for got, ref in zip(solve(items, precond), fresh[precond]):
            assert got[:2] == ref[:2]
            assert np.array_equal(got[2], ref[2]) and np.array_equal(got[3], ref[3])


def test_nonlinear_solve_after_a_failed_call():
    """The first search direction is written over whatever the work array holds (NaN here)."""
    p = W.cube_problem(16, 2.5, 1, "sin")
    p.g = np.where(p.chi_gamma > 0, 0.2 * W.random_field(p.nbox, 4), 0.0)
    r, g = torch.as_tensor(p.r, device=DEV), torch.as_tensor(p.g, device=DEV)
    H = rk.Handle.from_problem(p, device=DEV)
    ref = H.solve_nonlinear(r, g, "cubic", 5.0, tol=1e-8, max_iter=20000)[0]
    H.close()
    H = rk.Handle.from_problem(p, device=DEV)
    with pytest.raises(rk.RKError):
        H.transient_implicit(torch.full_like(r, float("nan")), g, 1e-3, 1, r.clone())
    got = H.solve_nonlinear(r, g, "cubic", 5.0, tol=1e-8, max_iter=20000)[0]
    assert torch.equal(got, ref)


def test_clone_does_not_wait_for_the_default_stream():
    """Work that the caller has in flight on the legacy default stream goes on."""
    p = W.cube_problem(32, 2.0, 1, "sin")
    H = rk.Handle.from_problem(p, device=DEV)
    H.clone().close()
    torch.cuda.synchronize()
    done = torch.cuda.Event()
    torch.cuda._sleep(int(2e9))  # about a second
    done.record()
    c = H.clone()
    assert not done.query()
    torch.cuda.synchronize()
    d = torch.as_tensor(W.random_field(p.nbox, 3), device=DEV)
    assert torch.equal(c.apply_K(d), H.apply_K(d))
