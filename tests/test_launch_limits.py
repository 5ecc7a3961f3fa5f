"""A kernel's launch attributes hold for one device, and a process may bind contexts on several, from several threads:
every attribute is set where a context is bound (the *_prepare functions, on the context's device), none on the way to
a launch behind a flag of the process."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_03430_gb300", "csrc")


def test_launch_attributes_are_set_at_bind():
    seen = 0
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        function = ""
        for n, line in enumerate(open(path), 1):
            m = re.match(r"[A-Za-z].*?(\w+)\([^;]*$", line)  # a definition starts in column 0
            if m:
                function = m.group(1)
            if "cudaFuncSetAttribute" in line:
                seen += 1
                assert "prepare" in function, f"{os.path.basename(path)}:{n} sets an attribute in {function}"
    assert seen >= 5
