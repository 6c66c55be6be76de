"""Kernels launched while their predecessor may still run (programmatic dependent
launch) must not tell the compiler that the memory they read is constant.

Read from the sources: such a kernel waits (griddepcontrol.wait), takes no
__restrict__ pointers, reads nothing that calls write through __ldg, and, where its
jobs lie in a table on the device, waits before it looks at the table.
"""
import os
import re

import paper_2609_02081_gb300 as hm

CSRC = os.path.join(os.path.dirname(os.path.abspath(hm.__file__)), "csrc")
WAIT = r"wait_for_previous_kernel\(\)|griddepcontrol\.wait"
UNITS = ["fp64_bilinear.cu", "split_gemm.cu", "split_kernels.cu", "split_mat2.cu"]


def source(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def functions(text):
    """(name, parameters, body) of the file's kernels and the device functions they call."""
    for m in re.finditer(r"__(?:global|device)__[^;{}()]*?(?:__launch_bounds__\([^)]*\)\s*)?(\w+)\s*\(", text):
        i, depth = m.end(), 1
        while depth:
            depth += {"(": 1, ")": -1}.get(text[i], 0)
            i += 1
        params, j = text[m.end():i - 1], text.find("{", i)
        if j < 0 or text[i:j].strip():
            continue
        k, depth = j + 1, 1
        while depth:
            depth += {"{": 1, "}": -1}.get(text[k], 0)
            k += 1
        yield m.group(1), params, text[j:k]


def waiting():
    return {(u, n): (p, b) for u in UNITS for n, p, b in functions(source(u)) if re.search(WAIT, b)}


def test_programmatic_kernels_wait():
    """Every kernel passed to launch_dependent waits for its predecessor."""
    launched = set()
    for u in UNITS:
        text = source(u)
        for m in re.finditer(r"launch_dependent\(", text):
            launched |= set(re.findall(r"\b(\w+_kernel)\b", text[m.end():m.end() + 260]))
        launched |= set(re.findall(r"\bgo\((\w+_kernel)", text))
    names = {n for _, n in waiting()}
    assert launched >= {"split_exponents_kernel", "mat2_encode_kernel", "split_residue_gemm_kernel", "mat2_crt_kernel",
                        "fp64_bilinear_kernel", "fp64_ranges_reduce_kernel"}
    assert launched <= names, launched - names


def test_programmatic_kernels_read_no_memory_as_constant():
    """No __restrict__ parameters and no __ldg, but of the module's own constants (g_m2digits, set up once per device);
    nor in the functions that hand the kernels their jobs."""
    found = waiting()
    assert len(found) >= 6
    for (u, n), (params, body) in found.items():
        assert "__restrict__" not in params, (u, n)
        assert not re.search(r"__ldg\((?!&g_m2digits\[)", body), (u, n)
        # intrinsics the compiler may move like arithmetic: through a pointer that exists only after the wait
        assert "__ldcg(" not in body or "known_from_here(" in body, (u, n)
    for u in ("split_device.cuh", "split_gemm.cu"):
        for n, params, body in functions(source(u)):
            if re.search(r"\bjobs\b", params):
                assert "__restrict__" not in params and "__ldg" not in body, (u, n)


def test_programmatic_kernels_wait_before_the_job_table():
    for (u, n), (params, body) in waiting().items():
        if not n.endswith("_kernel"):
            continue
        wait = re.search(WAIT, body).start()
        for use in re.finditer(r"\bunit_job\(|\bfind_item_job\(|\bfind_job\(|\bjobs\[", body):
            assert wait < use.start(), (u, n, use.group(0))


def test_launch_rules_use_the_devices_sm_count():
    """No rule of a launch compares with one chip's SM count (152) or its multiples."""
    for u in sorted(os.listdir(CSRC)):
        text = re.sub(r"/\*.*?\*/", "", source(u), flags=re.S)
        assert not re.findall(r"\b(?:152|304|608|1216)\b", text), u
