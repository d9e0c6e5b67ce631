"""Host memory that an asynchronous copy to the device reads outlives the call:
that such a copy has staged pageable memory when it returns is not promised, so
no copy starts from a container that dies with its scope."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2604_09113_gb300", "csrc")


def test_no_asynchronous_copy_from_a_local_container():
    seen = 0
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        src = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"cudaMemcpyAsync\(", src):
            depth, i = 1, m.end()
            while depth:
                depth += {"(": 1, ")": -1}.get(src[i], 0)
                i += 1
            call = src[m.end():i - 1]
            if "HostToDevice" not in call:
                continue
            seen += 1
            assert ".data()" not in call, (os.path.basename(path), call)
    assert seen >= 2
