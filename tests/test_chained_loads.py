"""Kernels that are launched programmatically live while the kernel before them
still writes their input, so they must not read it through the read-only path
(__ldg, const __restrict__): its loads are for data that nothing writes
meanwhile, and may be moved above the wait.  Checked in the source: which reads
of these functions go through it."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2008_11520_gb300", "csrc")

# function -> the buffers an earlier kernel of the chain writes
CHAINED = {
    "gru.cu": {"k_gru_rt": {"X"}},
    "stencil.cu": {
        "stage_padded": {"xcp"}, "own_patch": {"d"}, "edge_patches": {"d"}, "run4": {"d"},
        "scatter_fast_tile": {"d", "xcp"}, "scatter_cta": {"d", "xcp"}, "k_scatter_avg": {"d", "xcp"},
        "rhs_march": {"vc"}, "rhs_big": {"vc"}, "k_rhs_march": {"vc"},
    },
    "mg.cu": {"k_mg_vanka": {"dx"}, "k_mg_fixed": {"dx"}},
}
# what they may read so: the mesh's tables and maps, fixed while it lives
CONSTANT = re.compile(r"^(reinterpret_cast<const \w+ \*>\()?(pm\b|g\.(patch_id|tile_flags|slow_tiles|feat_tab)\b)")


def function(src, name):
    """(parameters, body) of the definition of a function."""
    at = re.search(r"\b%s\(" % name, src)
    assert at, name
    depth, i = 1, at.end()
    while depth:
        depth += {"(": 1, ")": -1}.get(src[i], 0)
        i += 1
    params = src[at.end():i - 1]
    j = src.index("{", i)
    depth, k = 1, j + 1
    while depth:
        depth += {"{": 1, "}": -1}.get(src[k], 0)
        k += 1
    return params, src[j:k]


@pytest.mark.parametrize("file,name", [(f, n) for f, d in CHAINED.items() for n in d])
def test_inputs_of_chained_kernels_are_read_coherently(file, name):
    with open(os.path.join(CSRC, file)) as f:
        params, body = function(f.read(), name)
    buffers = CHAINED[file][name]
    for b in buffers:
        p = [q for q in re.split(r",(?![^<]*>)", params) if re.search(r"\b%s$" % b, q.strip())]
        assert len(p) == 1, (name, b)
        assert "__restrict__" not in p[0], f"{name}: {p[0].strip()}"
    for arg in re.findall(r"__ldg\((.*)", body):
        assert CONSTANT.match(arg), f"{name}: __ldg({arg}"


def test_every_chained_launch_is_covered():
    """Kernels given to launch_chained read their inputs by TMA or are listed above."""
    tma = {"k_rhs", "k_restrict", "k_residual_step", "k_rhs_batch_small", "k_rhs_batch_march", "k_restrict_batch",
           "k_scatter_avg_batch"}   # (the batch forms call the listed functions)
    listed = {n for d in CHAINED.values() for n in d}
    for file in ("gru.cu", "stencil.cu"):
        with open(os.path.join(CSRC, file)) as f:
            src = f.read()
        for call in re.finditer(r"launch_chained\(\w+, (\w+)", src):
            k = call.group(1)
            if not k.startswith("k_"):   # a variable: the kernels assigned to it in this function
                start = src.rfind("\ntemplate ", 0, call.start())
                names = set(re.findall(r"\bk = (k_\w+)", src[start:call.start()]))
            else:
                names = {k}
            assert names and names <= listed | tma, (file, call.group(0), names)
