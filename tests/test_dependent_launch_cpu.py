"""Kernels that may be set up while the one before them runs (they start with follow()): what an
earlier kernel of a cycle writes is not read through a const __restrict__ parameter, which the
compiler may load before the wait. Read from the sources."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2103_11962_gb300", "csrc")

# written by no kernel that is launched this way: geometry, masks, index arrays, coefficients
# (with their flag and diagonal) and transfer weights, all of them the setup's, which ends in a
# synchronisation, and the caller's matrix
CONSTANT = {
    "coef", "half", "asym", "mult", "dinv", "c2", "slots", "gslot", "fregions", "cregions",
    "cmask", "cmult", "fmask", "wr", "gid", "affine", "rowptr", "col", "val", "regions", "c2r",
    "cgrp", "gptr", "rid",
}


def _kernels():
    """(name, parameter list, body) of every __global__ function."""
    for f in sorted(os.listdir(CSRC)):
        if not f.endswith((".cu", ".cuh")):
            continue
        src = open(os.path.join(CSRC, f)).read()
        src = re.sub(r"//[^\n]*", "", src)
        macro = re.search(r"#define RMG_SPLIT_PARAMS((?:[^\n]*\\\n)*[^\n]*)", src)
        if macro:
            src = src.replace("RMG_SPLIT_PARAMS) {", macro.group(1).replace("\\", " ") + ") {")
        for m in re.finditer(r"__global__\s+void\s+(?:__launch_bounds__\([^)]*\)(?:\s*,)?\s*)?"
                             r"(k_\w+)\(([^{]*)\)\s*\{", src):
            yield m.group(1), m.group(2), src[m.end():m.end() + 200]


def test_every_kernel_waits_before_anything_else():
    seen = 0
    for name, _, body in _kernels():
        if "follow(" in body:
            assert re.match(r"\s*follow\([\w, ]*\);", body), name
            seen += 1
    assert seen >= 20


def test_no_changing_data_behind_const_restrict():
    for name, params, body in _kernels():
        if not re.match(r"\s*follow\(", body):
            continue
        for p in params.split(","):
            m = re.search(r"const\s+\w[\w: ]*\*\s*__restrict__\s+(\w+)", p)
            if m:
                assert m.group(1) in CONSTANT, (name, m.group(1))
