"""Chained kernels (csrc/chain.cuh) may start before the kernels whose results they read have ended: no load
may move above the wait that opens them.  A __restrict__ pointer tells the compiler that nothing else,
the wait included, changes what it points to, so chained kernels take none (no GPU needed: this reads the
sources)."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2602_13841_gb300", "csrc")


def chained_kernels():
    """{name: parameter list} of the kernels that wait for the one before (chain_begin, chain_wait)."""
    out = {}
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        src = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"__global__\b.*?\b(k_\w+)\s*\(", src, flags=re.S):
            depth, i = 1, m.end()
            while depth:
                depth += {"(": 1, ")": -1}.get(src[i], 0)
                i += 1
            body = src[i:].lstrip()
            if body.startswith("{") and re.search(r"chain_(begin|wait)\(\)", body[:body.index("\n}")]):
                assert re.match(r"chain_(begin|wait)\(\);", body[1:].lstrip()), m.group(1)
                out[m.group(1)] = src[m.end():i - 1]
    return out


def test_chained_kernels_take_no_restrict_pointers():
    found = chained_kernels()
    assert {"k_cells2d", "k_cells3d", "k_node_sum", "k_vanka_stream", "k_transfer", "k_coarse_mv", "k_axpby",
            "k_dots", "k_sub_comb"} <= set(found)
    assert [name for name, params in found.items() if "__restrict__" in params] == []
