"""Order of the library's device work, read from its sources.

A caller's stream need not be ordered with the legacy default stream, so every launch and every
copy or clear of device memory names its stream.
"""

import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1004_5076_gb300", "csrc")


def _sources():
    for f in sorted(os.listdir(CSRC)):
        if f.endswith((".cu", ".cuh")):
            yield f, re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, f), encoding="utf-8").read())


def test_every_launch_and_clear_names_its_stream():
    for f, src in _sources():
        assert not re.findall(r"\bcudaMemset\w*(?<!Async)\s*\(", src), f
        for args in re.findall(r"<<<(.*?)>>>", src, re.S):
            depth, commas = 0, 0
            for ch in args:
                depth += ch in "([{"
                depth -= ch in ")]}"
                commas += ch == "," and depth == 0
            assert commas == 3, (f, args)


def test_every_copy_names_its_stream():
    for f, src in _sources():
        assert not re.findall(r"\bcudaMemcpy\w*(?<!Async)\s*\(", src), f


def _functions(src):
    """(name, parameters, body) of every function with a body."""
    for m in re.finditer(r"\b(?!if|for|while|switch)(\w+)\s*\(([^(){};]*)\)\s*\{", src):
        end, depth = m.end(), 1
        while depth:
            depth += {"{": 1, "}": -1}.get(src[end], 0)
            end += 1
        yield m.group(1), m.group(2), src[m.end():end]


# What an early-launched kernel may read by the read-only path: set-up tables, and vectors that
# were complete before the kernel's direct predecessor started.
TABLES = {"gp", "gpoff", "gpl", "gpr", "gpe", "gq", "xw", "acol", "acoord", "tw", "tw1", "tw2", "tw64", "ghE", "ghI",
          "gtE", "gtI", "mE", "mI", "nmv", "nmt", "gval", "pinv", "eunk"}
COMPLETE = {"k_rows": {"x"}, "k_rows_adj": {"y"}, "k_bdots": {"V"}, "k_bvsub_norm": {"V"}}


def test_early_launched_kernels_read_their_predecessor_by_plain_loads():
    kernels, readers = {}, set()
    for f, src in _sources():
        for name, params, body in _functions(src):
            if "pdl_wait();" in body:
                read_only = {p.split()[-1] for p in params.split(",") if "const" in p and "__restrict__" in p}
                kernels[name] = read_only - TABLES - COMPLETE.get(name, set())
            if "__ldg(" in body:
                readers.add((name, re.sub(r"\s+", " ", params.split(",")[0])))
    assert {"k_project", "k_axis0", "k_axis0_pm", "k_planes64", "k_rows", "k_bdots", "k_bvsub_norm"} <= set(kernels)
    assert not any(kernels.values()), kernels
    # the other users of __ldg: tables, and kernels that start after their predecessor's end
    assert {n for n, _ in readers} == {"load_group", "load4", "load_two", "load_desc", "ldg_cx", "k_point_fields"}
    assert {p for n, p in readers if n == "load_two"} == {"const float* p", "const double* p"}
    for f, src in _sources():
        assert set(re.findall(r"\bldg_cx\((?!const)\*?(\w+)", src)) <= {"M"}, f
