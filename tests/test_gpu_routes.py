"""Which way an operator goes -- direct sums or transform passes -- where the support allows
both, and that both give the same.  Tolerances as in the other parity tests: FP64 1e-10, FP32
2e-6; two solves to a residual of 1e-11 agree in u to 1e-8 (the smallest modes of K that u sees lie
a factor of some hundreds below its largest).
"""
import numpy as np
import pytest

from oracle.oracle import apply_K_sampled
from paper_2403_19854_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2403_19854_gb300 import rk  # noqa: E402

DEV = torch.device("cuda:0")


def tdev(x):
    return torch.as_tensor(np.ascontiguousarray(x), device=DEV)


def used_passes(H, call, prec):
    H.profile(True)
    call()
    torch.cuda.synchronize()
    seen = H.profile_read()
    H.profile(False)
    return ("x_merge", prec) in seen


def steps(H, p, prec):
    return H.solve(tdev(p.r), tdev(p.g), precision=prec, tol=1e-14, max_iter=4, want_u=False, raise_on_error=False)


# box, support, degree: are K in FP32 and in FP64, the FP32 part of a CG step, U^T taken by passes?
# (None: either way, their times are within a few percent of each other)
ROUTES = [((256, 256, 256), 2.5, 1, (False, False, True, False)), ((128, 128, 128), 1.5, 1, (False, False, False, False)),
          ((96, 96, 96), 2.5, 1, (False, False, False, False)), ((144, 144, 144), 3.5, 1, (False, False, True, False)),
          ((64, 64, 64), 4.5, 2, (False, True, None, True)), ((128, 128, 128), 4.5, 2, (None, None, True, True)),
          ((96, 96, 96), 4.5, 1, (False, True, None, False)), ((128, 128, 128), 4.5, 1, (False, True, None, None)),
          ((144, 144, 144), 4.5, 1, (False, None, None, False))]


@pytest.mark.parametrize("box,a,deg,want", ROUTES, ids=lambda v: str(v).replace(" ", ""))
def test_routes(box, a, deg, want):
    p = W.cube_problem(box[0], a, deg, "sin")
    H = rk.Handle.from_problem(p, device=DEV)
    d = tdev(W.random_field(p.nbox, 3))
    got = (used_passes(H, lambda: H.apply_K(d.float()), "f32"), used_passes(H, lambda: H.apply_K(d), "f64"),
           used_passes(H, lambda: steps(H, p, "mixed"), "f32"),
           used_passes(H, lambda: H.rhs(d), "f64"))
    for k, (g, w) in enumerate(zip(got, want)):
        assert w is None or g == w, (k, got, want)
    H.close()


@pytest.mark.parametrize("box,a,deg", [((64, 64, 64), 4.5, 1), ((64, 64, 64), 4.5, 2), ((96, 100, 64), 4.5, 1),
                                       ((162, 64, 72), 4.5, 2), ((128, 36, 144), 4.5, 2)])
def test_both_ways_agree(box, a, deg):
    """While a first call is captured the direct sums serve (the passes need workspaces made
    ahead); later calls of these boxes go by passes."""
    p = W.embed(W.cube_problem(min(box), a, deg, "sin"), box)
    H = rk.Handle.from_problem(p, device=DEV)
    d = tdev(np.where(p.chi > 0, W.random_field(p.nbox, 5), np.nan))
    d32 = d.float()
    out = [torch.empty_like(d), torch.empty_like(d), torch.empty_like(d32)]
    warm = rk.Handle.from_problem(p, device=DEV)  # (sets the kernels' attributes)
    for f, x in ((warm.apply_K, d), (warm.rhs, d), (warm.apply_K, d32)):
        f(x)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        H.apply_K(d, out[0])
        H.rhs(torch.nan_to_num(d), out[1])
        H.apply_K(d32, out[2])
    graph.replay()
    torch.cuda.synchronize()
    ref = [H.apply_K(d), H.rhs(torch.nan_to_num(d)), H.apply_K(d32)]
    for got, want, tol in zip(out, ref, (1e-10, 1e-10, 2e-6)):
        assert float((got - want).abs().max()) <= tol * float(want.abs().max())
    H.close()


@pytest.mark.parametrize("box,a,deg", [((144, 128, 162), 4.5, 1), ((100, 128, 144), 3.5, 2), ((64, 64, 64), 4.5, 2),
                                       ((72, 64, 96), 4.5, 2)])
def test_passes_match_the_oracle(box, a, deg):
    """K at nodes on and off the boundary, in both precisions, by whichever way."""
    p = W.embed(W.spheres_problem(n_box=min(box), n_spheres=6, a_tilde=a, degree=deg, r_range=(0.2, 0.3), seed=5), box)
    H = rk.Handle.from_problem(p, device=DEV)
    rng = np.random.default_rng(1)
    sample = np.unique(np.concatenate([rng.choice(np.flatnonzero(p.chi), 30, replace=False),
                                       rng.choice(np.flatnonzero(p.chi_gamma), 20, replace=False)]))
    d = W.random_field(p.nbox, 9)
    for dt, tol in ((np.float64, 1e-10), (np.float32, 2e-6)):
        x = d.astype(dt)
        f = H.apply_K(tdev(x)).cpu().numpy().astype(np.float64)
        ref = apply_K_sampled(p.n, p.h, a, deg, p.chi, p.V, x.astype(np.float64) * p.chi, sample)
        assert np.abs(f[sample] - ref).max() <= tol * np.abs(ref).max()
        assert np.all(f[p.chi == 0] == 0.0)
    H.close()


@pytest.mark.parametrize("box", [(256, 128, 144)], ids=str)
def test_mixed_solve_with_wide_supports(box):
    """The FP32 CG steps of a box above 128^3 nodes with r = 2 (by passes) against the FP64 solve."""
    p = W.embed(W.cube_problem(min(box), 2.5, 1, "sin"), box)
    p.g = np.where(p.chi_gamma > 0, 0.1, 0.0)
    H = rk.Handle.from_problem(p, device=DEV)
    assert used_passes(H, lambda: steps(H, p, "mixed"), "f32")
    us = [H.solve(tdev(p.r), tdev(p.g), precision=prec, tol=1e-11)[1] for prec in ("mixed", "fp64")]
    assert float((us[0] - us[1]).abs().max()) <= 1e-8 * float(us[1].abs().max())
    H.close()
