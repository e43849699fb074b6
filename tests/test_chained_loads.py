"""Kernels that may start while the launch before them still runs (those that
call grid_dependency) read what that launch writes by ordinary loads: __ldg
wants data that nothing writes while the kernel lives.  Read from the sources;
__ldg is left to the kernels below, whose reads are older than the launch
before them."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1203_1269_gb300", "csrc")

OLDER = {
    "k_assemble_tiles": "the caller's theta",
    # the double factor; k_rhs_f64, k_fit_finish or k_residual_vec lies between
    "k_fwd_diag_f64": "factor", "k_fwd_tiles_f64": "factor", "k_bwd_diag_f64": "factor", "k_bwd_tiles_f64": "factor",
    # the split factor; k_fwd_diag lies between
    "k_fwd_tiles": "factor",
}


def chained_kernels():
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"__global__[^{;]*?\b(k_\w+)\s*\([^{;]*\)\s*\{", text):
            depth, i = 1, m.end()
            while depth:
                depth += {"{": 1, "}": -1}.get(text[i], 0)
                i += 1
            body = text[m.end():i]
            if "grid_dependency();" in body:
                yield m.group(1), body


def test_ldg_only_on_older_data():
    kernels = dict(chained_kernels())
    assert len(kernels) >= 30 and set(OLDER) <= set(kernels)
    for name, body in kernels.items():
        assert body.lstrip().startswith("grid_dependency();"), name
        assert "__ldg(" not in body or name in OLDER, name
