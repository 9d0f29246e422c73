"""Kernels launched with programmatic stream serialisation (csrc/adjoint.cu, launch_after) start while the kernel that
writes their inputs still runs: neither they nor the device functions they call may have their reads marked as
read-only for the kernel's life (__restrict__ on a pointer to const, __ldg, ld.global.nc)."""
import os
import re

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_astro_ph_0702058_gb300", "csrc")


def _functions(text):
    """name -> text from its parameter list to its closing brace, of every function that has a body."""
    out = {}
    for m in re.finditer(r"\b(\w+)\s*\(", text):
        depth, k = 1, m.end()
        while depth and k < len(text):
            depth += {"(": 1, ")": -1}.get(text[k], 0)
            k += 1
        body = re.match(r"\s*(const\s*)?\{", text[k:])
        if not body or m.group(1) in ("if", "for", "while", "switch"):
            continue
        end, depth = k + body.end(), 1
        while depth and end < len(text):
            depth += {"{": 1, "}": -1}.get(text[end], 0)
            end += 1
        out[m.group(1)] = text[m.start():end]
    return out


def test_no_read_only_loads_of_the_previous_kernels_output():
    code = "".join(open(os.path.join(SRC, f)).read() for f in
                   ("ptx.cuh", "force_x2.cuh", "step_impl.cuh", "adjoint.cu"))
    functions = _functions(re.sub(r"//[^\n]*", "", code))
    kernels = [n for n, t in functions.items() if "after_previous();" in t]
    assert sorted(kernels) == ["adj_step_kernel", "roll_step_kernel", "vjp_pairs_kernel"]
    reached, todo = set(), list(kernels)
    while todo:
        name = todo.pop()
        if name in reached:
            continue
        reached.add(name)
        todo += [w for w in set(re.findall(r"\b\w+\b", functions[name])) if w in functions]
    assert {"vjp_at_slot", "column_sums", "vjp_pair", "vjp_fold", "corr_dim"} <= reached
    for name in sorted(reached):
        assert not re.search(r"__restrict__|__ldg|ld\.global\.nc", functions[name]), name
