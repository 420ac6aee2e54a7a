"""Outputs that share memory with an input: f^q written over q or over A (or both, q == A), in
one, two and three dimensions, on boxes of one and of many blocks.  The same sums of the same
values as with arrays of their own: 1e-14 of the largest value covers another order of the
products.
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

PROBLEMS = [lambda: W.line_problem(64, 2.5, 1), lambda: W.plane_problem(16, 2.5, 1), lambda: W.plane_problem(256, 3.0, 2),
            lambda: W.cube_problem(16, 1.5, 1, "zero"), lambda: W.cube_problem(36, 4.5, 1, "zero"),
            lambda: W.cube_problem(100, 2.5, 1, "zero"), lambda: W.cube_problem(48, 3.0, 2, "zero")]


@pytest.mark.parametrize("k", range(len(PROBLEMS)))
def test_boundary_rhs_over_its_inputs(k):
    p = PROBLEMS[k]()
    H = rk.Handle.from_problem(p, device=DEV)
    rng = np.random.default_rng(k)
    q = torch.as_tensor(rng.standard_normal(p.nbox), device=DEV)
    A = torch.as_tensor(np.where(p.chi_gamma > 0, rng.uniform(0.5, 1.5, p.nbox), 0.0), device=DEV)
    ref = H.boundary_rhs(q, A)
    both = H.boundary_rhs(A, A)
    tol = 1e-14

    def same(f, g):
        assert float((f - g).abs().max()) <= tol * float(g.abs().max())

    for _ in range(5):
        x = A.clone()
        same(H.boundary_rhs(q, x, out=x), ref)
        x = q.clone()
        same(H.boundary_rhs(x, A, out=x), ref)
        x = A.clone()
        same(H.boundary_rhs(x, x, out=x), both)
    # a weight that overlaps the output in part
    n = p.nbox
    buf = torch.empty(2 * n, dtype=torch.float64, device=DEV)
    off = (n // 2) // 2 * 2
    w, f = buf[:n], buf[off:off + n]
    w.copy_(A)
    same(H.boundary_rhs(q, w, out=f), ref)
    H.close()
