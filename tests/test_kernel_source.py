"""What the device code may not contain, read from its source."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2608_00867_b200", "csrc")


def device_code():
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        with open(path) as f:
            for number, line in enumerate(f, 1):
                yield f"{os.path.basename(path)}:{number}", line.split("//")[0]


def test_no_non_coherent_loads():
    """A kernel behind a programmatic launch runs while its predecessor still writes the sources: they are not read-only
    for the kernel's lifetime, which ld.global.nc (and __ldg, and loads the compiler derives from const __restrict__) ask."""
    found = [at for at, code in device_code() if re.search(r"\bld\.global(\.\w+)*\.nc\b|__ldg\b|__restrict__", code)]
    assert not found, found
