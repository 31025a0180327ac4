"""Kernels that are set up while the kernel before them still runs (they call step_begin()) read memory which that kernel
writes.  A load that the compiler may take for read-only (a `const ... __restrict__` parameter, __ldg) is not ordered by the
wait in step_begin(), so neither occurs in such a kernel or in a device function that it calls.  The constant tables of
load_tables64() are read-only for good."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2002_03644_gb300", "csrc")
HEAD = re.compile(r"(?:__global__|__device__)[^;{}()]*?(?:__launch_bounds__\([^)]*\)\s*)?\b(\w+)\s*\(([^;{}]*)\)\s*(?:const\s*)?\{")
READ_ONLY = re.compile(r"\bconst\b[^,]*\*\s*__restrict__")


def functions():
    """name -> list of (parameters, body) of every device function and kernel of the step."""
    out = {}
    for f in sorted(os.listdir(CSRC)):
        if not f.endswith(".cuh"):
            continue
        src = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, f)).read())
        for m in HEAD.finditer(src):
            depth, at = 1, m.end()
            while depth:
                depth += {"{": 1, "}": -1}.get(src[at], 0)
                at += 1
            out.setdefault(m[1], []).append((m[2], src[m.end():at]))
    return out


FUNCTIONS = functions()
CHAINED = sorted(k for k, v in FUNCTIONS.items() if any("step_begin()" in body for _, body in v))


def test_the_chained_kernels_are_found():
    assert {"fused_step_kernel", "march_pair_kernel", "march_moment_kernel", "split_level_kernel", "split_collide_kernel",
            "wall_ghost_kernel"} <= set(CHAINED)


@pytest.mark.parametrize("kernel", CHAINED)
def test_no_read_only_load_of_the_state(kernel):
    seen, todo = set(), [kernel]
    while todo:
        name = todo.pop()
        if name in seen or name == "load_tables64":
            continue
        seen.add(name)
        for params, body in FUNCTIONS[name]:
            assert not READ_ONLY.search(params), (name, params)
            assert "__ldg(" not in body, name
            todo += [w for w in set(re.findall(r"\b(\w+)\s*(?:<[^;{}()]*>)?\(", body)) if w in FUNCTIONS]
