"""Copies onto the device are ordered with the kernels that read them: the library's streams do not
wait for the legacy stream, on which cudaMemcpy from pageable memory may return before the data is on
the device (and from device memory before it has begun).  So every such copy, and every fill, names a stream."""
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1407_3868_gb300", "csrc")


def test_copies_onto_the_device_name_a_stream():
    seen = 0
    for name in sorted(os.listdir(CSRC)):
        if not name.endswith((".cu", ".cuh", ".cpp", ".h")):
            continue
        with open(os.path.join(CSRC, name)) as f:
            text = f.read()
        for call in re.findall(r"cudaMemcpy\([^;]*?cudaMemcpy(\w+)\)", text):
            assert call == "DeviceToHost", (name, call)
            seen += 1
        assert not re.search(r"cudaMemset\(", text), name
    assert seen > 0
