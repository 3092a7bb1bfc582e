"""Kernels that may start while the kernel before them still runs (they wait for it on the
device) read what that kernel writes.  CUDA defines the read-only load path, which __ldg and
const __restrict__ pointers take, only for data that nothing writes while the kernel runs, so
none of them may use it.  A race of this kind depends on scheduling; it is checked in the
sources (no GPU)."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2607_08186_gb300", "csrc")


def _closing(src, at, pair):
    depth = 0
    for i in range(at, len(src)):
        depth += (src[i] == pair[0]) - (src[i] == pair[1])
        if depth == 0:
            return i
    raise AssertionError("unbalanced source")


def _kernels():
    """(name, parameter list, body) of every kernel."""
    out = []
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        src = re.sub(r"//[^\n]*|/\*.*?\*/", "", open(path).read(), flags=re.S)
        for m in re.finditer(r"__global__\s+void\s+(?:__\w+__\s*\([^()]*\)\s*)*(\w+)\s*\(", src):
            end = _closing(src, m.end() - 1, "()")
            start = src.index("{", end)
            out.append((os.path.basename(path) + ":" + m.group(1), src[m.end():end],
                        src[start:_closing(src, start, "{}") + 1]))
    return out


def _early():
    return [k for k in _kernels() if re.search(r"\b(grid|attn)_dep_wait\s*\(", k[2])]


def test_the_early_kernels_are_found():
    names = {k[0].split(":")[1] for k in _early()}
    assert {"fwd_kernel", "fwd256_kernel", "bwd_kernel", "bwd256_kernel", "sfa_bwd_prep_kernel", "dkv_finalize_kernel",
            "decode_kernel", "decode_tc_kernel", "combine_kernel", "append_kernel", "expand_embed_kernel", "rank_kernel",
            "scatter_kernel", "rows_kernel", "select_kernel", "select_bwd_kernel"} <= names


@pytest.mark.parametrize("name,params,body", _early(), ids=[k[0] for k in _early()])
def test_no_read_only_loads(name, params, body):
    for p in params.split(","):
        assert not ("__restrict__" in p and re.search(r"\bconst\b[^*]*\*", p)), p.strip()
    assert "__ldg" not in body
