"""Overlapped launches begin while their predecessor still writes populations, so the read-only path
(ld.global.nc, __ldg) may serve only what no kernel of a march writes: the force field and a batch's tile table."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_0809_4730_gb300", "csrc")


def test_read_only_path_serves_constant_data_only():
    calls = 0
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        for line in open(path):
            code = line.split("//")[0]
            assert "ld.global.nc" not in code, (path, line)
            for arg in re.findall(r"__ldg\((.*)", code):
                calls += 1
                generic = "void ldgv(const float* p" in code          # the force field of one or two nodes
                assert generic or re.match(r"(a|b)\.Ffield|tile_start", arg), (path, line)
            for arg in re.findall(r"\bldgv\((?!const)([^,]*),", code):
                assert arg.startswith("b.Ffield"), (path, line)
    assert calls > 0
