"""Kernels that may start while their predecessor drains (programmatic
dependent launch) read what an earlier kernel wrote behind their wait, through
pointers that are not __restrict__: the qualifier lets the compiler use the
read-only path and move the loads ahead of the wait.  Checked on the sources:
in these kernels, and in the device functions of their vectors, __restrict__
marks only data that no kernel of the cycle (or of the factorisation) writes."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2103_07537_gb300", "csrc")
SRC = {f: open(os.path.join(CSRC, f)).read() for f in sorted(os.listdir(CSRC)) if f.endswith((".cu", ".cuh"))}

# matrices, patterns, index maps and inverses: written by the setup alone
CONSTANT = {"rp", "ci", "vals", "lowk", "upk", "agg", "agg_ptr", "members", "ainv", "inv", "lu", "diag", "row_sys",
            "node_off", "inv_off", "Xq"}
VECTORS = {"x", "x_in", "xt", "uc", "rhs", "rf", "y", "xp", "res"}


def dependent_kernels():
    names = {"coarse_cycle_kernel"}
    for text in SRC.values():
        names |= set(re.findall(r"launch_k\((\w+_kernel)\b", text))
        names |= set(re.findall(r"launch_pdl\(\(const void\*\)(\w+)", text))
    return sorted(names)


def closing(text, i, pair):
    """Index behind the bracket that closes the one before i."""
    depth = 1
    while depth:
        depth += {pair[0]: 1, pair[1]: -1}.get(text[i], 0)
        i += 1
    return i


def definition(name):
    """(parameters, body) of a kernel's definition."""
    for text in SRC.values():
        for m in re.finditer(r"\b%s\s*\(" % name, text):
            i = closing(text, m.end(), "()")
            if "__global__" in text[max(0, m.start() - 160):m.start()] and text[i:].lstrip().startswith("{"):
                return text[m.end():i], text[i:closing(text, text.index("{", i) + 1, "{}")]
    raise AssertionError(name)


def restrict_names(code):
    return set(re.findall(r"__restrict__\s+(\w+)", code))


def test_the_kernels_are_found():
    names = set(dependent_kernels())
    assert len(names) >= 20 and {"spmv_tpr_kernel", "gs_inner_kernel", "tc_panel_kernel"} <= names


@pytest.mark.parametrize("name", dependent_kernels())
def test_vectors_are_not_restrict(name):
    params, body = definition(name)
    assert restrict_names(params) | restrict_names(body) <= CONSTANT


def test_device_functions_of_the_vectors():
    for f in ("bgs_body.cuh", "k_solve.cu", "k_coarse.cu"):
        for m in re.finditer(r"__device__[^;{]*\(([^{;]*)\)\s*\{", SRC[f]):
            assert restrict_names(m.group(1)) <= CONSTANT | {"vb"}, (f, m.group(0))  # vb: a row of the matrix


def test_rows_loaded_as_constant_are_matrix_rows():
    for f, text in SRC.items():
        for arg in re.findall(r"load_row<[^>]*>\((\w+)", text):
            assert arg not in VECTORS, (f, arg)
