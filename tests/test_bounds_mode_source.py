"""The bounds mode (-DEMB_CHECK) covers the kernels that index by values from data: each of these
functions checks its index with emb_ck before the access."""
from __future__ import annotations

import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2512_01251_gb300", "csrc")

CHECKED = {  # file: {function: checks at least}
    "emb_internal.cuh": {"emb_lookup": 2},
    "emb_common.cu": {"nbr_row3": 2},
    "emb_refine.cu": {"in": 1},
    "emb_bin.cu": {"k_filter_list": 1},
    "emb_voxelize.cu": {"vox_line": 1},
    "emb_forest.cu": {"k_make_children": 4},
    "emb_cutlinks.cu": {"k_link_cand": 1, "k_link_lists": 1, "k_link_emit": 2},
    "emb_lbm.cu": {"k_lbm_step": 1},
    "emb_splice.cu": {"k_sp_place": 1, "k_sp_bits": 1, "k_sp_rank": 2, "k_sp_link_counts": 1, "k_sp_link_copy": 1},
    "emb_backward.cu": {"k_qbwd_tile": 2, "k_qbwd_scatter": 1},
}


def _body(src, name):
    """The braces of the first definition of `name`."""
    for m in re.finditer(rf"\b{name}\s*\(", src):
        depth, i = 1, m.end()
        while depth:
            depth += {"(": 1, ")": -1}.get(src[i], 0)
            i += 1
        rest = re.match(r"\s*(const)?\s*\{", src[i:])
        if not rest:
            continue
        start = i = i + rest.end()
        depth = 1
        while depth:
            depth += {"{": 1, "}": -1}.get(src[i], 0)
            i += 1
        return src[start:i]
    raise AssertionError(f"no definition of {name}")


@pytest.mark.parametrize("file", list(CHECKED))
def test_indices_from_data_are_checked(file):
    src = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, file)).read())
    for name, least in CHECKED[file].items():
        assert _body(src, name).count("emb_ck(") >= least, name


def test_every_access_to_the_refine_bitmap_is_checked():
    src = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, "emb_refine.cu")).read())
    for name in ("test", "clear", "row"):
        body = _body(src, name)
        assert "in(p" in body and body.index("in(p") < body.index("w[p >>" if "w[p >>" in body else "atomicAnd")
