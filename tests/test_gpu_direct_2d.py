"""The direct sums on 2D boxes at every support they take (one to four nodes to a side), both
bases: K in both precisions, u^h, U^T and f^r against the oracle, on boxes whose sides leave
partial tiles and with the domain across the periodic boundary.  Tolerances as in the other
parity tests (FP64 1e-10, FP32 2e-6).
"""
import numpy as np
import pytest

from oracle.oracle import Oracle
from paper_2403_19854_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2403_19854_gb300 import rk  # noqa: E402

DEV = torch.device("cuda:0")


def tdev(x):
    return torch.as_tensor(np.ascontiguousarray(x), device=DEV)


@pytest.mark.parametrize("box,shift", [((36, 48), (30, 5)), ((162, 64), (1, 60)), ((100, 72), (0, 0))], ids=str)
@pytest.mark.parametrize("a,deg", [(1.5, 1), (2.5, 1), (3.5, 1), (4.5, 1), (3.0, 2), (3.5, 2), (4.5, 2)])
def test_plane_operators(box, shift, a, deg):
    p = W.embed(W.plane_problem(min(box), a, deg), box + (1,))
    o = Oracle(p.n, p.h, a, deg, p.chi)

    def roll(v):
        return np.roll(v.reshape(box[1], box[0]), (shift[1], shift[0]), axis=(0, 1)).reshape(-1)

    H = rk.Handle(p.n, p.h, tdev(roll(p.chi)), tdev(roll(p.chi_gamma)), tdev(roll(p.V)), deg, a)
    m = roll(p.chi) > 0
    d = W.random_field(p.nbox, 3)
    dc = d * p.chi

    def close(got, ref, tol, what):
        got = got.cpu().numpy().astype(np.float64)
        assert np.abs(got - roll(ref))[m].max() <= tol * np.abs(ref).max(), what
        assert np.all(got[~m] == 0.0), what

    noisy = np.where(m, roll(d), np.nan)
    close(H.apply_K(tdev(noisy)), o.apply_K(p.V, dc), 1e-10, "K FP64")
    d32 = d.astype(np.float32)
    close(H.apply_K(tdev(noisy.astype(np.float32))), o.apply_K(p.V, d32.astype(np.float64) * p.chi), 2e-6, "K FP32")
    close(H.eval_u(tdev(roll(d))), o.eval_u(dc), 1e-10, "u^h")
    close(H.eval_u_transpose(tdev(roll(d))), o.eval_u_transpose(dc), 1e-10, "U^T")
    close(H.rhs(tdev(roll(d))), o.rhs(p.V, dc), 1e-10, "f^r")
    H.close()
