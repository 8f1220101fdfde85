"""Kernels launched as dependent ones overlap the kernel before them, and read-only loads (__ldg,
ld.global.nc, const __restrict__) are defined only for memory that nothing writes during a kernel's
lifetime: in these kernels, and the device functions among them, they may read only what no kernel of a
solve writes.  A reading of the source: no run on a GPU has shown a stale value."""

import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1704_08897_gb300", "csrc")

# written by the host, or by kernels that no dependent one follows directly
CONSTANT = {"slots", "tcp", "items", "n_items", "gate",            # descriptors, work lists (gate: a volatile read)
            "S.lamx", "S.lamy", "&S.wnorm", "S.low_qyd", "qx_h", "qx_l", "g.B", "Bl",  # eigenvalues, bases
            "reinterpret_cast<const char*>(&S)",                   # the descriptor itself
            "mask", "b"}                                           # the 3-D solve's mask and right-hand side


def functions(name):
    """(head, body) of every function of the file."""
    src = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())
    for m in re.finditer(r"^(?:template <[^\n]*>\n)?(?:static )?(?:__global__|__device__)[^;{]*\{", src, re.M):
        line = src[m.end():src.index("\n", m.end())]
        end = m.end() + len(line) if line.rstrip().endswith("}") else src.index("\n}", m.end())
        yield src[m.start():m.end()], src[m.end():end]


@pytest.mark.parametrize("name", ["kernels_grid.cu", "kernels_gemm_tc.cu", "solve3d.cu"])
def test_dependent_kernels_read_only_constants_as_read_only(name):
    seen = 0
    for head, body in functions(name):
        if "__global__" in head and "pdl_wait()" not in body and "gate_shut(" not in body and "stencil_producer" not in body:
            continue  # launched in full order
        seen += 1
        for arg in re.findall(r"(?:__ldg|ld_early|ld_keep)\(((?:[^()]|\([^()]*\))*)\)", body):
            if not arg.startswith("const "):  # (the helpers' own heads)
                assert arg.split(" + ")[0].strip() in CONSTANT, (head.split("(")[0], arg)
        for var in re.findall(r"\bconst \w+ ?\*? ?\*\s*(?:const )?__restrict__ (\w+)", head + body):
            assert var in CONSTANT, (head.split("(")[0], var)
    assert seen > 5
