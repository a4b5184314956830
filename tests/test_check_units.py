"""Every unit with kernels has an index-check counter that mcg_bounds_violations adds up (read from the sources)."""
import os
import re

from paper_0807_0264_gb300 import build

TEXT = {u: open(os.path.join(build.CSRC, u)).read() for u in build.SOURCES}


def test_units_with_kernels_are_counted():
    total = TEXT["mcg_capi.cu"].split("long long mcg_bounds_violations", 1)[1].split("#else", 1)[0]
    for unit, text in TEXT.items():
        if "__global__" not in text:
            continue
        reader = re.search(r"MCG_BOUND_READER\((\w+)\)", text)
        assert reader, f"{unit} has kernels and no counter"
        assert f"{reader.group(1)}(r)" in total, f"{unit}: its counter is not added up"
