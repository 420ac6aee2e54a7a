"""The CG steps fused into the operator kernels, step by step: a fixed number of them from
the same start, against the same steps formed from the operator on its own, and again and
again with the same bits.

Tolerances: six steps of CG lose no more than a few digits to the order of the sums: FP64
1e-10.  In FP32 each of the six A p, p . A p and updates carries a few roundings of 6e-8, and
alpha and beta pass them on: 1e-4.
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
STEPS = 6


def problem(box, a, deg):
    p = W.embed(W.cube_problem(min(box), a, deg, "sin"), box)
    rng = np.random.default_rng(7)
    # data on every node of the domain, so that a wrong value anywhere shows
    p.r = np.where(p.chi > 0, rng.standard_normal(p.nbox), 0.0)
    p.g = np.where(p.chi_gamma > 0, 0.1, 0.0)
    return p


def cg(H, p, steps):
    """x on the free nodes after `steps` of CG in FP64 from the operators of the handle."""
    t = lambda x: torch.as_tensor(x, device=DEV)  # noqa: E731
    free = t(((p.chi > 0) & (p.chi_gamma == 0)).astype(np.float64))
    g = t(p.g)
    r = free * (H.rhs(t(p.r)) - H.apply_K(g))
    x, q, rr = torch.zeros_like(r), r.clone(), torch.dot(r, r)
    for _ in range(steps):
        Aq = free * H.apply_K(q)
        al = rr / torch.dot(q, Aq)
        x, r = x + al * q, r - al * Aq
        new = torch.dot(r, r)
        q, rr = r + (new / rr) * q, new
    return x


# boxes whose CG steps run in the regular stencil, in blocks of nodes and in the walk of every
# node; sides that leave partial tiles, rows that are no multiple of 16 bytes, every reach
CASES = [((128, 128, 128), 1.5, 1, "mixed"), ((162, 96, 100), 2.0, 1, "mixed"), ((128, 100, 144), 1.5, 1, "fp64"),
         ((162, 96, 100), 2.5, 1, "fp64"), ((96, 128, 100), 3.0, 2, "fp64"), ((128, 96, 128), 4.5, 1, "fp64"),
         ((36, 162, 48), 2.5, 1, "mixed"), ((162, 36, 48), 3.5, 1, "mixed"), ((48, 36, 32), 4.5, 1, "mixed"),
         ((162, 128, 144), 2.5, 1, "mixed"), ((144, 128, 162), 3.0, 2, "mixed"), ((100, 162, 1), 2.5, 1, "fp64")]


@pytest.mark.parametrize("box,a,deg,prec", CASES, ids=lambda v: str(v).replace(" ", ""))
def test_fused_steps(box, a, deg, prec):
    if box[2] == 1:
        p = W.embed(W.plane_problem(min(box[:2]), a, deg), box)
        p.r = np.where(p.chi > 0, np.random.default_rng(7).standard_normal(p.nbox), 0.0)
    else:
        p = problem(box, a, deg)
    check(p, prec)


@pytest.mark.parametrize("box,a,deg,prec", [((162, 96, 100), 1.5, 1, "mixed"), ((162, 36, 48), 2.5, 1, "mixed"),
                                            ((48, 36, 32), 4.5, 1, "mixed"), ((64, 72, 64), 2.5, 1, "fp64"),
                                            ((72, 100, 128), 3.0, 2, "fp64")], ids=lambda v: str(v).replace(" ", ""))
def test_fused_steps_across_the_periodic_boundary(box, a, deg, prec):
    p = problem(box, a, deg)
    shift = (box[2] - 3, box[1] // 2, 5)
    for k in ("chi", "chi_gamma", "V", "r", "g"):
        setattr(p, k, np.roll(getattr(p, k).reshape(box[2], box[1], box[0]), shift, axis=(0, 1, 2)).reshape(-1))
    check(p, prec)


def check(p, prec):
    H = rk.Handle.from_problem(p, device=DEV)
    ref = cg(H, p, STEPS).cpu().numpy()
    r, g = torch.as_tensor(p.r, device=DEV), torch.as_tensor(p.g, device=DEV)
    first = None
    for _ in range(12):
        d, _, info = H.solve(r, g, precision=prec, tol=1e-14, max_iter=STEPS, want_u=False, raise_on_error=False)
        assert info["iterations"] == STEPS
        d = d.cpu().numpy()
        if first is None:
            first = d
        assert np.array_equal(d, first), "the same steps with other bits"
    e = np.abs(first - p.g - ref).max() / np.abs(ref).max()
    assert e < (1e-10 if prec == "fp64" else 1e-4), e
    H.close()
