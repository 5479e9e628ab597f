"""Which kernels the debug build's index checks reach, read from the sources:
every kernel that steps a batch or takes several steps per launch names a
site of csrc/bounds.cuh in the code that forms its addresses."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1107_4543_gb300", "csrc")
SITES = {"step_multi.cuh": {"rows_task": "ROWS_NODE", "k_rows_batch": "BATCH_REC",
                            "k_step_tile": "TILE_NODE"},
         "resident.cuh": {"k_batch_resident": "RES_NODE", "k_resident_tiny": "RES_NODE",
                          "resident_load": "RES_NODE", "resident_store": "RES_NODE"},
         "step_impl.cuh": {"step_task": "BATCH_LANE", "batch_block": "BATCH_REC"}}


def body(src, name):
    """The text of function `name` from its parameter list to its last brace."""
    at = re.search(r"\b%s\(const" % name, src) or re.search(r"\b%s\(T \*" % name, src)
    i = src.index("{", src.index(") {", at.start()))
    depth = 0
    for k in range(i, len(src)):
        depth += (src[k] == "{") - (src[k] == "}")
        if depth == 0:
            return src[i:k]
    raise AssertionError(name)


def test_kernels_name_their_check_sites():
    for name, sites in SITES.items():
        with open(os.path.join(CSRC, name)) as f:
            src = re.sub(r"//[^\n]*", "", f.read())
        for fn, site in sites.items():
            assert "bounds::" + site in body(src, fn), (name, fn)
