"""No asynchronous copy to the device reads a host variable by its address: the copy may still be running when
the variable's scope ends (pageable memory is read by the device itself on hardware-coherent systems)."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2402_02075_gb300", "csrc")


def test_no_asynchronous_copy_from_a_local_variable():
    found = []
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        text = open(path).read()
        for m in re.finditer(r"cudaMemcpyAsync\([^;]*?cudaMemcpy(HostToDevice|Default)[^;]*;", text, re.S):
            if re.match(r"cudaMemcpyAsync\([^,]+,\s*&", m.group(0)):
                found.append(f"{os.path.basename(path)}: {' '.join(m.group(0).split())}")
    assert not found, found
