"""Kernels that are launched to overlap the kernel before them read vectors only
after the wait: no vector goes through a read-only load or a __restrict__
pointer, which the code generator may move above it.  Read from the source (no
GPU needed); what may be read early are the tables that no kernel writes."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2305_15116_gb300", "csrc")

# names of tables written at set-up only: stencils, work lists, incidences,
# coordinates, inverse diagonals, the dense level-0 inverse
TABLES = {"w", "wd", "wf", "wk", "mi", "row", "incs", "ic", "prims", "items", "v_items", "e_items", "tiles", "rec",
          "ab", "d", "f", "hi", "lo", "h1", "l1", "dinv", "dv", "lpts", "v_of_slot", "slot_of_v"}
# face_weights' table; the policies' load, which only P2's row takes
EXTRA = {"iface3d.cuh": {"p"}, "arith.cuh": {"p"}}
# functions of kernels that are launched after everything before them has finished
PLAIN = {"multigrid.cu": ("k_diag_part", "k_diag_iface", "k_diag_invert"),
         "p2.cu": ("row", "p2_boundary_point", "k_p2_rows")}
# every launch of these files is of that kind
FILES = sorted(f for f in os.listdir(CSRC) if f.endswith((".cu", ".cuh")) and f not in ("problem.cu", "noalloc.cu"))


def _overlapped(name):
    src = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())
    for fn in PLAIN.get(name, ()):
        src, n = re.subn(r"(__device__|__global__)[^;{}]*\b" + fn + r"\(.*?\n}\n", "", src, count=1, flags=re.S)
        assert n == 1, fn
    return src


@pytest.mark.parametrize("name", FILES)
def test_vectors_are_read_after_the_wait(name):
    src = _overlapped(name)
    tables = TABLES | EXTRA.get(name, set())
    bad = [m.group(0) for m in re.finditer(r"\*\s*__restrict__\s+(\w+)", src) if m.group(1) not in tables]
    for m in re.finditer(r"__ldg\(((?:[^()]|\([^()]*\))*)\)", src):
        arg = re.sub(r"(static|reinterpret)_cast<[^>]*>", "", m.group(1))
        base = re.match(r"\W*([\w.\->]+?)\W*(?:[ +)]|$)", arg).group(1)
        if re.split(r"\.|->", base)[-1] not in tables:
            bad.append(m.group(0))
    if name != "p2.cu" and "P::load(" in src:
        bad.append("P::load")
    assert not bad, bad
