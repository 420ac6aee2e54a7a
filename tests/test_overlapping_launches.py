"""Kernels that may overlap the kernel before them (grid_wait) read what that one writes: such
data must not go through the read-only path, which requires it to stay unchanged for the whole
kernel.  Checked in the sources: no __restrict__ parameter, and no __ldg of a CG step's vectors.
"""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2403_19854_gb300", "csrc")


def kernels():
    """(file, name, parameters, body) of every __global__ function."""
    for f in sorted(os.listdir(CSRC)):
        src = open(os.path.join(CSRC, f)).read()
        for m in re.finditer(r"__global__[^;{]*?\b(k_\w+)\(", src):
            at, depth = m.end(), 1
            while depth:
                depth += {"(": 1, ")": -1}.get(src[at], 0)
                at += 1
            params = src[m.end():at]
            if src[at:].lstrip()[:1] != "{":
                continue
            start = src.index("{", at)
            end, depth = start + 1, 1
            while depth:
                depth += {"{": 1, "}": -1}.get(src[end], 0)
                end += 1
            yield f, m.group(1), params, src[start:end]


def test_no_read_only_loads_of_data_in_flux():
    waiting = [k for k in kernels() if "grid_wait()" in k[3]]
    assert {k[1] for k in waiting} >= {"k_cg_xr_fused", "k_cell_sums", "k_cell_spread", "k_regular", "k_delta", "k_correct"}
    for f, name, params, body in waiting:
        assert "__restrict__" not in params, f"{f}: {name}"
        assert not re.search(r"__ldg\((a\.)?(p_old|p_new|p0|p1|gall|delta|out)\b", body), f"{f}: {name}"
        # the input of a CG step is the residual that the update before it writes: __ldg(a.in)
        # stands in the branch of a plain operator only
        for m in re.finditer(r"__ldg\(a\.in\b", body):
            before = body[:m.start()]
            plain = before.rfind("} else {") > before.rfind("if constexpr (CG)") >= 0
            assert plain or "Alg. 4: g_p = b0_p y" in before, f"{f}: {name}"
