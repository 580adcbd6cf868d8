"""The library keeps no state in function-local variables: what is set per device or per object would
otherwise be taken as set by other devices, objects and threads."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2412_13402_gb300", "csrc")


def test_no_function_keeps_a_mutable_static_variable():
    files = glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh"))
    assert len(files) > 8
    found = []
    for path in files:
        for n, line in enumerate(open(path), 1):
            # an indented `static T name = ...` or `static T name;` (not a constant, not a member function)
            if re.match(r"\s+static\s+(?!const\b|constexpr\b)[^()/]*[=;]", line):
                found.append(f"{os.path.basename(path)}:{n}: {line.strip()}")
    assert not found, found
