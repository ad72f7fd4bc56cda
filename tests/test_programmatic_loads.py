"""Kernels launched with programmatic stream serialization are resident while the launch before still writes
the fields they read: those reads must be ordinary loads.  The read-only path (ld.global.nc) is specified for
memory that nothing writes during the kernel, and the compiler may move such a load above
griddepcontrol.wait.  A replay that happens to be right cannot show this, so the sources are checked: in every
file with a programmatic kernel, field loads are the ordinary form and only links are read by __ldg."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1106_4964_gb300", "csrc")


def test_programmatic_kernels_read_fields_by_ordinary_loads():
    files = [f for f in glob.glob(os.path.join(CSRC, "*.cu*")) if "pdl_wait()" in open(f).read()]
    assert len(files) >= 3
    for f in files:
        text = re.sub(r"//[^\n]*", "", open(f).read())
        for call in re.findall(r"\b(?:load_spinor|load_spinor_unscaled)<([^>]*)>", text):
            assert call.replace(" ", "").endswith(",false"), (f, call)
        for call in re.findall(r"\bld_field<([^>]*)>", text):
            assert call == "false", (f, call)
        for arg in re.findall(r"__ldg\(([^\n]*)", text):
            assert arg.startswith("lb "), (f, arg)  # links
