"""Every kernel of the library that derives node indices from its launch coordinates and takes the place of a
checked one on a default path tests its index ranges in the checked build, and its translation unit's record
is read.  By the sources: the kernel's own text or the text of a function that only it calls."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1903_12522_gb300", "csrc")
CHECK = re.compile(r"CMCG_RANGE_OK|column_in_range|chunk_in_range|plane_map\(|plane_it\(|Column<DIM> m\(")


def text_of(source, name):
    """The function's text: from its name's definition to the brace in column 0."""
    m = re.search(r"\b" + name + r"\([^;{]*\)[^;{]*\{", source, re.S)
    assert m, name
    return source[m.start():source.index("\n}\n", m.start())]


@pytest.mark.parametrize("file,names", [
    ("step_row.cu", ["k_step_row"]), ("step_band.cu", ["k_band", "k_band4"]), ("step_block.cu", ["k_block3"]),
    ("step_soft.cu", ["k_step_soft", "k_start_soft", "k_end_soft", "k_adj_prep_soft", "k_adj_start_soft", "k_adj_final_soft",
                      "k_pcg_applyK", "k_pcg_cluster"]),
    ("first_order.cu", ["k_fo_row", "k_fo_row_load", "k_fo_row_end"]),
    ("riesz.cu", ["k_coarse_vcycle", "neighbour_sum", "at", "k_mg3_first", "k_mg2_first"]),
])
def test_kernel_tests_its_indices(file, names):
    source = open(os.path.join(CSRC, file)).read()
    unit = re.search(r"CMCG_CHECK_TU\((\w+)\)", source)
    assert unit, file
    assert f"check_read_{unit.group(1)}" in open(os.path.join(CSRC, "api.cu")).read()
    for name in names:
        assert CHECK.search(text_of(source, name)), name
