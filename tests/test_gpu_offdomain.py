"""Values off the domain are ignored (K d and u^h read chi o d, f^r reads r on chi), where the
operators run as transform passes and as direct sums: NaN there gives the bits of zeros there.
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

# supports wider than the direct sums take, in one, two and three dimensions, and narrower ones
PROBLEMS = [lambda: W.line_problem(64, 5.5, 1), lambda: W.plane_problem(36, 5.5, 1), lambda: W.plane_problem(100, 6.0, 2),
            lambda: W.cube_problem(32, 5.5, 1), lambda: W.embed(W.cube_problem(36, 5.5, 2), (162, 36, 48)),
            lambda: W.embed(W.cube_problem(32, 5.5, 1), (100, 32, 36)),
            lambda: W.plane_problem(36, 2.5, 1), lambda: W.plane_problem(100, 4.5, 2), lambda: W.cube_problem(16, 1.5, 1),
            lambda: W.embed(W.cube_problem(32, 2.5, 1), (100, 32, 36)), lambda: W.cube_problem(48, 3.0, 2),
            lambda: W.cube_problem(100, 2.5, 1), lambda: W.cube_problem(64, 4.5, 2)]


@pytest.mark.parametrize("k", range(len(PROBLEMS)))
def test_nan_off_the_domain(k):
    p = PROBLEMS[k]()
    H = rk.Handle.from_problem(p, device=DEV)
    m = torch.as_tensor(p.chi > 0, device=DEV)
    d = torch.as_tensor(W.random_field(p.nbox, 3), device=DEV)
    zero, nan = torch.where(m, d, 0.0), torch.where(m, d, float("nan"))
    for f in (H.apply_K, H.eval_u, H.rhs, lambda x: H.apply_K(x.float())):
        ref, got = f(zero), f(nan)
        assert bool(torch.isfinite(ref).all())
        assert torch.equal(got, ref)
    H.close()


@pytest.mark.parametrize("a,deg", [(2.0, 1), (4.5, 1), (5.5, 1)])
def test_solve_reads_the_source_on_the_domain(a, deg):
    p = W.cube_problem(32, a, deg, "sin")
    H = rk.Handle.from_problem(p, device=DEV)
    r = torch.as_tensor(p.r, device=DEV)
    nan = torch.where(torch.as_tensor(p.chi > 0, device=DEV), r, float("nan"))
    kw = dict(precision="fp64", tol=1e-30, max_iter=20, raise_on_error=False)
    ref, got = H.solve(r, **kw), H.solve(nan, **kw)
    assert got[2]["status"] == ref[2]["status"] and got[2]["iterations"] == 20
    assert torch.equal(got[0], ref[0]) and torch.equal(got[1], ref[1])
    H.close()
