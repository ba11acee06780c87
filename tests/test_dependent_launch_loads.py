"""A kernel launched as a programmatic dependent is resident while the kernel before it may still be writing
its inputs.  The non-coherent load path asks for data that is constant for the kernel's whole life, and the compiler may
move such loads across griddepcontrol.wait.  So no kernel that waits there reads through it: neither by __ldg /
ld.global.nc nor by parameters that promise read-only, unaliased data (on a pointer that is only read,
__restrict__ is that promise)."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1910_02120_b200", "csrc")
WAIT = re.compile(r"pdl_wait\(\)|griddepcontrol\.wait")


def _sources():
    for f in sorted(os.listdir(CSRC)):
        if f.endswith((".cu", ".cuh", ".h")):
            text = open(os.path.join(CSRC, f)).read()
            yield f, re.sub(r"//[^\n]*", "", text)


def _closing(text, at, pair):
    depth = 0
    for i in range(at, len(text)):
        depth += (text[i] == pair[0]) - (text[i] == pair[1])
        if depth == 0:
            return i
    raise AssertionError("unbalanced " + pair)


def _kernels(text):
    """(name, parameter list, body) of every __global__ function that is defined."""
    for m in re.finditer(r"__global__", text):
        head = re.compile(r"(\w+)\s*\(").search(text, m.end())
        while head.group(1).startswith("__"):           # __launch_bounds__(...), __cluster_dims__(...)
            head = re.compile(r"(\w+)\s*\(").search(text, _closing(text, head.end() - 1, "()"))
        end = _closing(text, head.end() - 1, "()")
        brace = text.find("{", end)
        if brace < 0 or ";" in text[end:brace]:
            continue
        yield head.group(1), text[head.end():end], text[brace:_closing(text, brace, "{}") + 1]


def test_kernels_are_found():
    waiting = [k for _, text in _sources() for k, _, body in _kernels(text) if WAIT.search(body)]
    assert len(waiting) >= 20 and {"gemm_f32_kernel", "gemm_short_kernel", "move_kernel", "rows_kernel", "permute_cols_kernel",
                                   "stage_rows_kernel", "eval_rows_wide_kernel", "gemm_tc_kernel"} <= set(waiting), waiting


def test_no_noncoherent_loads():
    found = [(f, n + 1) for f, text in _sources() for n, line in enumerate(text.split("\n"))
             if re.search(r"__ldg\s*\(|ld\.global\.nc", line)]
    assert not found, found


def test_inputs_of_waiting_kernels_are_not_restrict():
    bad = []
    for f, text in _sources():
        for name, params, body in _kernels(text):
            if not WAIT.search(body):
                continue
            for p in params.split(","):
                if "__restrict__" not in p:
                    continue
                var = re.search(r"(\w+)\s*$", p).group(1)
                # written through in every instance: not under a template switch between the directions
                if "const" in p or name in ("rows_kernel", "permute_cols_kernel") and var != "opw":
                    bad.append((f, name, var))
    assert not bad, bad
