"""Kernels launched as programmatic dependents may be resident while the kernel
before them still writes their operands, so they must not read those through
the read-only path: not by __ldg, and not through a const __restrict__ parameter
(which the compiler may read that way).  That path is for the plan's tables.
Checked on the sources of every kernel that waits by grid_wait."""
import glob
import os
import re

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1711_11296_gb300", "csrc")

# Read-only for a transform's whole life: the P~ table and pointers into it,
# its row exponents, problem and tile lists, first nodes, FFT tables.
TABLE_PARAMS = {"pnm", "probs", "tiles", "jmin"}
TABLE_POINTERS = {"P", "A", "pe", "eap", "tw", "A.rev"}


def _kernels():
    """(file, name, parameters, body) of every kernel or kernel body that waits."""
    out = []
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.h"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"\b(\w+(?:_kernel|_body))\(([^;{}]*?)\)\s*\{", text):
            depth, i = 1, m.end()
            while depth:
                depth += {"{": 1, "}": -1}.get(text[i], 0)
                i += 1
            body = text[m.end():i]
            if re.search(r"\bgrid_wait\(|\bbegin_fft\(", body):
                out.append((os.path.basename(path), m.group(1), m.group(2), body))
    return out


KERNELS = _kernels()


def test_the_dependent_kernels_are_found():
    names = {k[1] for k in KERNELS}
    assert {"slice_b_kernel", "slice_gemm_kernel", "split_b_kernel", "split_gemm_body",
            "legendre_small_fp64_kernel", "fx_forward_kernel", "fft_inverse_kernel"} <= names


@pytest.mark.parametrize("path,name,params,body", KERNELS, ids=["%s:%s" % k[:2] for k in KERNELS])
def test_reads_of_other_kernels_results(path, name, params, body):
    for p in re.findall(r"const\s+[\w<>]+\s*\*\s*__restrict__\s+(\w+)", params):
        assert p in TABLE_PARAMS, p
    for arg in re.findall(r"__ldg\(\s*([\w.]+)", body):
        assert arg in TABLE_POINTERS, arg


def test_device_functions_of_the_ffts():
    # (called by the kernels above; their operands come as structs)
    for fn in ("sht_fft64.cu", "sht_fft_kernels.h"):
        text = open(os.path.join(CSRC, fn)).read()
        for arg in re.findall(r"__ldg\(\s*([\w.]+)", text):
            assert arg in TABLE_POINTERS, (fn, arg)
