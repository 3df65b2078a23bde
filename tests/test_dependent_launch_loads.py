"""A kernel that starts by programmatic dependent launch lives while the one before it still writes.
The read-only path (__ldg, ld.global.nc) is for data that nothing writes during the kernel's life, so in
the sources of such kernels it reads constant tables only."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2209_14889_gb300", "csrc")


@pytest.mark.parametrize("source", ["lb3d.cu", "lb_conv.cu", "lb_unet.cu", "lb_diffuse.cu", "lb_diffuse.cuh", "lb_node.cuh",
                                    "lb_cell.cuh", "lb_tile.cuh", "lb_fused.cu"])
def test_read_only_loads_are_of_tables_only(source):
    src = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, source)).read())
    assert not [m for m in re.findall(r"__ldg\(([^;]*?)\)", src) if "lut" not in m and "(L" not in m]     # lut, L: the tables
    assert "global.nc" not in src and not re.findall(r"__restrict__ (?!L\b|lut)\w+", src)
