"""Every CUDA runtime call whose failure would leave wrong tables, descriptors or launch
limits behind is checked: in the sources of the library's own paths no copy, fill,
synchronisation, attribute or device query stands as a statement with its result dropped.
(An error of an upload that goes unseen turns up as wrong numbers, not as HEOM_ECUDA.)"""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2601_20550_gb300", "csrc")
FILES = ["api.cu", "batched.cu", "checkpoint.cu", "f64_stage.cu", "grad.cu", "internal.h", "kernels.cu", "noalloc.cu",
         "steady.cu"]
CALLS = r"cuda(Memcpy\w*|Memset\w*|StreamSynchronize|DeviceSynchronize|FuncSetAttribute|GetDevice|DeviceGetAttribute|LaunchKernelEx)"


@pytest.mark.parametrize("name", FILES)
def test_no_dropped_result(name):
    src = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())
    # a call is a statement of its own if it follows ; { } : or the ) of an if or for
    dropped = [m.group(1) for m in re.finditer(r"(?:^|[;{}:)])\s*(" + CALLS + r"\s*\([^;]*;)", src)]
    assert not dropped, dropped
