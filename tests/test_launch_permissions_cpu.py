"""A launch's permission for more than 48 KB of shared memory belongs to the
device that was current when it was asked for, so nothing in the sources may
remember per process that it was: no flag of static storage, and the attribute
is set in allow_shared (each launch that needs it) or where a batch's plan is
uploaded (per device) only."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2109_14340_gb300", "csrc")


def test_no_permission_is_remembered():
    setters = {}
    for name in sorted(os.listdir(CSRC)):
        if not name.endswith((".cu", ".cuh")):
            continue
        with open(os.path.join(CSRC, name)) as f:
            text = f.read()
        assert not re.search(r"\bstatic\s+bool\s+\w+\s*=", text), name
        n = len(re.findall(r"\bcudaFuncSetAttribute\(", text))
        if n:
            setters[name] = n
    assert setters == {"teno_dev.cuh": 1, "teno_batch.cu": 2}
