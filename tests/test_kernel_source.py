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


def host_functions():
    """(where, text) of every function of the host code, cut at the lines that start in the first column."""
    with open(os.path.join(CSRC, "nuna_api.cu")) as f:
        for text in re.split(r"\n(?=[a-z])", re.sub(r"//.*", "", f.read())):
            yield text.split("\n", 1)[0], text


def test_device_tables_are_not_set_behind_the_streams_back():
    """cudaMemset, and cudaMemcpy out of pageable memory, return before they are done, and only the legacy stream and those that
    wait for it come after them: control words, flags and work lists, which a kernel on any other stream may use next, cannot
    be set that way.  The measuring hooks launch on the legacy stream itself."""
    found = [at for at, text in host_functions() if "nuna_debug_" not in at and
             re.search(r"\bcudaMemset\(|\bcudaMemcpy\([^;]*HostToDevice", text)]
    assert not found, found
