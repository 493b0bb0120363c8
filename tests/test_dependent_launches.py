"""Memory ordering of dependent launches, from the CUDA sources (no GPU).

A kernel launched with programmatic stream serialization exists while the
kernel before it still writes; what that kernel wrote may be read after
griddepcontrol.wait, and only by ordinary loads: the read-only path (__ldg,
ld.global.nc, const __restrict__ pointers) is for memory that stays constant
for the life of the kernel, and the compiler may move such loads above the
wait.
"""
import os
import re

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2512_01032_gb300", "csrc")
READ_ONLY = re.compile(r"__ldg|__ldcs|__ldlu|__ldcv|\bld_ro\b|ld\.global\.nc|ld\.global\.\w*\.?nc|"
                       r"__restrict__|tex1D")


def _code():
    txt = ""
    for f in sorted(os.listdir(CSRC)):
        if f.endswith((".cu", ".cuh")):
            txt += open(os.path.join(CSRC, f)).read() + "\n"
    txt = re.sub(r"//[^\n]*", "", txt)
    return re.sub(r"/\*.*?\*/", "", txt, flags=re.S)


def _functions(code):
    """name -> text (signature and body) of every device function and kernel;
    overloads and specialisations of a name are joined."""
    out = {}
    for m in re.finditer(r"(__global__|__device__)[^;{}]*?\b(\w+)\s*\((?=[^;{}]*\{)", code):
        # the name is the identifier before the parameter list
        head = code[m.start():code.index("{", m.end())]
        head = re.sub(r"__launch_bounds__\s*\((?:[^()]|\([^()]*\))*\)|__maxnreg__\s*\([^()]*\)", "",
                      head)
        name = re.search(r"\b(\w+)\s*\(", head).group(1)
        k, depth = code.index("{", m.end()), 0
        for e in range(k, len(code)):
            depth += {"{": 1, "}": -1}.get(code[e], 0)
            if depth == 0:
                break
        out[name] = out.get(name, "") + head + code[k:e + 1]
    return out


def _launched_dependently(code):
    """Kernels passed to launch_dependent(), directly or by expression."""
    return set(re.findall(r"launch_dependent\(\s*(\w+)", code)) - {"void"}


CODE = _code()
FUNCS = _functions(CODE)
KERNELS = sorted(_launched_dependently(CODE))


def test_every_waiting_kernel_is_covered():
    assert {"k_phase1", "k_phase2", "k_read_phi", "k_read_cell", "k_batch_phase1",
            "k_batch_phase2", "k_diag_fold"} <= set(KERNELS)
    for name, body in FUNCS.items():
        waits = re.search(r"\blaunch_ready\s*\(\s*\)\s*;", body) is not None
        assert waits == (name in KERNELS) or name == "launch_ready", name
    assert CODE.count("ProgrammaticStreamSerialization") == 1  # launch_dependent() alone
    assert {"gather_g", "ld_h_cell", "xbc_cell", "finish_cell", "store_cell"} <= set(FUNCS)


@pytest.mark.parametrize("kernel", KERNELS)
def test_no_read_only_loads_under_a_dependent_launch(kernel):
    seen, todo = set(), [kernel]
    while todo:
        f = todo.pop()
        if f in seen:
            continue
        seen.add(f)
        hit = READ_ONLY.search(FUNCS[f])
        assert not hit, f"{kernel} reaches {hit.group(0)} in {f}"
        todo += [g for g in set(re.findall(r"\b(\w+)\s*(?=[(<])", FUNCS[f])) if g in FUNCS]


def test_a_waiting_kernel_touches_no_memory_before_the_wait():
    """launch_ready() is the first statement (declarations of shared memory
    and compile-time constants aside)."""
    for k in KERNELS:
        body = FUNCS[k][FUNCS[k].index("{") + 1:]
        for st in body.split(";"):
            st = st.strip()
            if st.startswith("launch_ready"):
                break
            assert st.startswith(("__shared__", "constexpr")), (k, st)
        else:
            raise AssertionError(k)
