"""Every translation unit whose kernels follow item ids or tile numbers read from memory takes part
in the bounds-checked build: it checks them with in_bounds and the context binds its bounds word."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2408_12677_gb300", "csrc")


def test_units_with_ids_from_memory_are_bound():
    api = open(os.path.join(CSRC, "api.cu")).read()
    for unit in ("raster", "tilebin", "prefix"):
        src = open(os.path.join(CSRC, unit + ".cu")).read()
        assert len(re.findall(r"in_bounds\(", src)) >= 2, unit
        assert re.search(unit + r"_bind_bounds\(uint32_t\* word\) \{ return bind_bounds_word\(word\); \}", src), unit
        assert unit + "_bind_bounds(c->d_bounds)" in api, unit
