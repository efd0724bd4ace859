"""What the kernels of a launch chain read, found in their source (no GPU needed).

A kernel that calls grid_dependency_wait() is resident while the kernel before it still
writes (csrc/internal.h, launch_chained).  `const __restrict__` and __ldg say that memory does
not change while the kernel lives, so they are for the caller's inputs only."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2608_14563_gb300", "csrc")
INPUTS = {"h", "w", "y", "W_U"}                    # kernel parameters that hold caller's inputs
LDG = {"p.y", "hr", "p.w", "wy", "pos.src(p.Y[g]"}  # __ldg operands that do (epilogues.cuh)
PLAIN = {"ld_row_raw"}                             # device functions of kernels launched plainly


def _sources():
    for name in sorted(os.listdir(CSRC)):
        if name.endswith((".cu", ".cuh")):
            with open(os.path.join(CSRC, name)) as f:
                yield name, re.sub(r"//[^\n]*", "", f.read())


def _functions(text):
    """(name, parameters, body) of every device function and kernel."""
    for m in re.finditer(r"__(?:global|device)__[^;{}]*?(\w+)\(((?:[^()]|\([^()]*\))*)\)"
                         r"(?:\s*const)?\s*\{", text):
        depth, i = 1, m.end()
        while depth:
            depth += {"{": 1, "}": -1}.get(text[i], 0)
            i += 1
        yield m.group(1), m.group(2), text[m.end():i]


def test_chained_kernels_read_results_with_ordinary_loads():
    kernels, bad = 0, []
    for file, text in _sources():
        for name, params, body in _functions(text):
            chained = "grid_dependency_wait()" in body
            kernels += chained
            is_kernel = re.search(r"__global__[^;{}]*\b%s\(" % name, text) is not None
            if (is_kernel and not chained) or name in PLAIN:
                continue  # launched plainly: starts when every kernel before has completed
            for p in re.findall(r"const\s[^,]*?\*\s*__restrict__\s+(\w+)", params):
                if p not in INPUTS:
                    bad.append("%s: %s reads %s as unchanging" % (file, name, p))
        if file == "epilogues.cuh":
            for m in re.finditer(r"__ldg\((?:reinterpret_cast<[^>]*>\()?([\w.]+(?:\(p\.\w+\[g\])?)",
                                 text):
                if m.group(1) not in LDG:
                    bad.append("%s: __ldg(%s)" % (file, m.group(1)))
    assert kernels >= 18  # the pattern still finds them
    assert not bad, bad
