"""Which kernels are loaded together: the driver loads a compilation unit as one when its first kernel is launched, so the kernels
that every path needs must not sit beside the many instances of a path of its own (source text only)."""
import os
import re

from paper_2309_13307_b200 import build


def kernels_of(source):
    text = open(os.path.join(build.CSRC, source)).read()
    return set(re.findall(r"__global__\s+void(?:\s+__launch_bounds__\([^)]*\))?\s+(\w+)\(", text))


def test_finishing_kernels_load_without_a_projection():
    home = [s for s in build.SOURCES if "finish_project_kernel" in kernels_of(s)]
    assert len(home) == 1
    assert kernels_of(home[0]) == {"finish_project_kernel", "finish_aggregate_kernel", "aggregate_kernel"}


def test_every_unit_is_built():
    assert sorted(build.SOURCES) == sorted(f for f in os.listdir(build.CSRC) if f.endswith(".cu"))
