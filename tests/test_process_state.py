"""A call leaves the process as it found it: nothing in the library sets an
attribute of a kernel or of the device, which every later call of the process
would see (its speed, or the grid that follows from occupancy, would depend on
what ran before)."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2004_04071_gb300", "csrc")


def test_no_kernel_or_device_attribute_is_set():
    sets = re.compile(r"\b(cu(?:da)?(?:FuncSet\w+|DeviceSet\w+|CtxSet(?!Current)\w+|KernelSet\w+))\s*\(")
    for name in sorted(os.listdir(CSRC)):
        if name.endswith((".cu", ".cuh", ".h")):
            with open(os.path.join(CSRC, name)) as fh:
                found = sets.findall(fh.read())
            assert not found, (name, found)
