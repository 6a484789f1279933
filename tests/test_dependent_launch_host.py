"""Kernels that may start before the one ahead of them has ended read through ordinary loads.

Such a kernel (launched by launch_dependent, waiting in after_previous) reads what the kernel
ahead wrote during its own lifetime, so neither a read-only load nor a __restrict__ pointer, which
lets the compiler choose one, may stand in it or in anything it calls.  Checked on the source text:
every kernel with after_previous() and the device functions it reaches."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2106_07694_gb300", "csrc")


def _functions():
    """name -> list of (qualifier, body) of the functions at namespace scope."""
    out = {}
    for f in sorted(os.listdir(CSRC)):
        if not f.endswith((".cu", ".cuh")):
            continue
        text = open(os.path.join(CSRC, f)).read()
        text = re.sub(r"//[^\n]*|/\*.*?\*/", "", text, flags=re.S)
        for m in re.finditer(r"^(?:__host__ )?(__device__|__global__)\b[^;{]*?\b(\w+)\(", text, re.M):
            name = m.group(2)
            if name == "__launch_bounds__":
                name = re.compile(r"\b(\w+)\(").search(text, text.index(") ", m.end())).group(1)
            at = text.find("{", m.end())
            depth, end = 0, at
            while True:
                depth += {"{": 1, "}": -1}.get(text[end], 0)
                end += 1
                if depth == 0:
                    break
            out.setdefault(name, []).append((m.group(1), text[m.start():end]))
    return out


def test_dependent_kernels_use_no_read_only_loads():
    fns = _functions()
    roots = [n for n, defs in fns.items() if any(q == "__global__" and "after_previous()" in b for q, b in defs)]
    assert {"rk_tile2d_kernel", "rk_stage2d_kernel", "rk_stage2d_wide_kernel", "lbm_d2q9_kernel",
            "lbm_d2q9_record_kernel", "sugar_kernel", "class_sum_kernel", "adj_stage_kernel",
            "adj_fluid_kernel"} <= set(roots)
    seen, todo, bad = set(), list(roots), []
    while todo:
        name = todo.pop()
        if name in seen:
            continue
        seen.add(name)
        for _, body in fns[name]:
            bad += [(name, w) for w in ("__restrict__", "__ldg", "LoadNC") if w in body]
            todo += [w for w in set(re.findall(r"\b\w+\b", body)) if w in fns]
    assert not bad


def test_every_dependent_launch_is_of_a_kernel_that_waits():
    fns = _functions()
    text = "".join(open(os.path.join(CSRC, f)).read() for f in os.listdir(CSRC) if f.endswith((".cu", ".cuh")))
    names = set(re.findall(r"launch_dependent\(\s*(?:lw::)?(\w+)[<(]", text))
    names = {"rk_tile2d_kernel" if n == "tile2d_entry" else "rk_stage2d_wide_kernel" if n == "stage2d_wide_entry" else n
             for n in names} - {"void"}
    assert len(names) >= 9
    for n in names:
        for _, body in fns[n]:
            assert re.search(r"\{\s*after_previous\(\);", body), n
